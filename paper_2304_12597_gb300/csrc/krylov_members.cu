// One Algorithm 2 per member of a batched plan.  K is block diagonal over the
// members (member b owns rows [b len, (b+1) len) and never couples to another), so
// each member runs the paper's Algorithm 2 on its own part b_b of b = sum_i gamma_i L_i
// (eq. 7): its own Krylov space K_m(K_b, b_b), Hessenberg T_m (eq. 10), capacitance
// system (eq. 12), residual estimate and stopping decision (eq. 13), exactly as if it
// were solved alone.  The members share the kernel launches, the stored shifted
// solves h_k and the basis array V (member b's entries in its own rows).
//
// A member's vectors are held in registers (len <= 8192 entries), by one thread-block cluster per
// member while the clusters of all members fit the SMs, else by one CTA: a vector step is FP64 work,
// and 512 threads on one SM per member left most SMs idle.  Measured per launch, init / Arnoldi /
// eq. (13), one CTA -> clusters:
//    8 members of 3969 rows  16.4 / 33.7 / 26.6 us -> 12.3 / 19.2 / 19.8 us (clusters of 8)
//    8 members of 2048 rows  14.3 / 22.8 / 16.4 us -> 12.3 / 15.3 / 16.3 us (of 8)
//   32 members of 1023 rows  14.3 / 16.8 / 16.3 us -> 12.2 / 15.3 / 18.3 us (of 4)
#include "pd_internal.h"
#include "pd_krylov.cuh"

namespace pd {

struct MemberView {
  double *scal;
  int *flags;
  double *T, *y;
  int64_t off;
};

__device__ __forceinline__ MemberView member_view(const KrylovBufs &k, int b) {
  MemberView v;
  v.scal = k.mscal + (int64_t)b * kScalWords;
  v.flags = k.mflags + (int64_t)b * kFlagWords;
  v.T = k.T + (int64_t)b * (k.maxit + 1) * k.maxit;
  v.y = k.y + (int64_t)b * (k.maxit + 1);
  v.off = (int64_t)b * k.mlen;
  return v;
}

// Batch totals after every member has finished a step (run by the last CTA):
// ||b|| and ||r_m|| as root sums of squares over the members, the loop flags, and the
// WHILE conditional (continue while any member runs).  start: after the first step.
// red: kRedWords doubles of shared memory.
__device__ void member_totals(const KrylovBufs &k, bool start, int use_handle, cudaGraphConditionalHandle h,
                              double *red) {
  __shared__ double out[2];
  double s[2] = {0.0, 0.0};
  int run = 0, conv = 1, nonfin = 0, zero = 1;
  for (int b = threadIdx.x; b < k.members; b += blockDim.x) {
    const double *sb = k.mscal + (int64_t)b * kScalWords;
    const int *fb = k.mflags + (int64_t)b * kFlagWords;
    s[0] += sb[S_BETA] * sb[S_BETA];
    s[1] += sb[S_RES] * sb[S_RES];
    run |= fb[F_KSTOP] ? 0 : 1;
    conv &= fb[F_KCONV] ? 1 : 0;
    nonfin |= fb[F_NONFIN] ? 1 : 0;
    zero &= fb[F_BZERO] ? 1 : 0;
  }
  run = __syncthreads_or(run);
  conv = __syncthreads_and(conv);
  nonfin = __syncthreads_or(nonfin);
  zero = __syncthreads_and(zero);
  block_sums(s, 2, red, out);
  if (threadIdx.x == 0) {
    double *scal = k.scal;
    int *flags = k.flags;
    if (nonfin) flags[F_NONFIN] = 1;
    scal[S_RES] = sqrt(out[1]);
    if (start) {
      scal[S_BETA] = sqrt(out[0]);
      scal[S_T] = 0.0;
      flags[F_BREAK] = 0;  // a member's breakdown only stops that member
      flags[F_BZERO] = zero;
      flags[F_CAPCNT] = 0;
      flags[F_M] = 0;
    } else {
      flags[F_M] += 1;
    }
    const bool stop = !run || nonfin || flags[F_M] >= k.maxit;
    flags[F_KSTOP] = stop ? 1 : 0;
    flags[F_KCONV] = conv;
    if (use_handle) cudaGraphSetConditional(h, stop ? 0u : 1u);
    *k.counter = 0;
  }
}

// Start of Algorithm 2 for member blockIdx.y: beta_b = ||b_b||, v_1 = b_b / beta_b, its
// T_m and y_m cleared, its control block reset.
template <int MODE, int E>
__global__ void __launch_bounds__(MODE == kCluster ? kBlasCluster : kBlasSingle) k_member_init(KrylovBufs k, const double *__restrict__ b,
                                                            int use_handle, cudaGraphConditionalHandle h) {
  grid_dep_wait();
  __shared__ double red[kRedWords];
  __shared__ double c[34];
  const MemberView mv = member_view(k, blockIdx.y);
  const int len = k.mlen;
  __shared__ double cslot[MODE == kCluster ? kSlot : 1];
  const int f = g_first<MODE>(), st = g_stride<MODE>();
  for (int i = f; i < (k.maxit + 1) * k.maxit; i += st) mv.T[i] = 0.0;
  for (int i = f; i <= k.maxit; i += st) mv.y[i] = 0.0;
  double x[E];
  reg_load<MODE, E>(len, b + mv.off, x);
  const double beta = sqrt(reg_norm2<MODE, E>(x, cslot, 0, red, c));
  const double ib = beta > 0.0 ? 1.0 / beta : 0.0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = f + e * st;
    if (j < len) {
      const double v = x[e] * ib;
      k.V[mv.off + j] = v;
      if (k.Vf) k.Vf[mv.off + j] = (float)v;
    }
  }
  if (g_leader<MODE>()) {
    const bool finite = isfinite(beta), zero = !(beta > 0.0);
    double *scal = mv.scal;
    int *flags = mv.flags;
    scal[S_BETA] = beta;
    scal[S_T] = 0.0;
    scal[S_RES] = beta;
    scal[S_HIST] = beta;
    flags[F_BREAK] = 0;
    flags[F_BZERO] = zero ? 1 : 0;
    flags[F_NONFIN] = finite ? 0 : 1;
    flags[F_CAPCNT] = 0;
    flags[F_M] = 0;
    flags[F_FROZEN] = 0;  // no step is frozen until an Arnoldi step says so (q > 1)
    flags[F_NOH] = 0;
    flags[F_KSTOP] = (finite && !zero) ? 0 : 1;
    flags[F_KCONV] = zero ? 1 : 0;
  }
  cluster_exit<MODE>();
  if (last_cta_done(k.counter)) member_totals(k, true, use_handle, h, red);
}

// One Arnoldi step (eq. 10) for member blockIdx.y, as in the single-problem kernel;
// a member that has stopped writes a zero row instead.
template <int MODE, int E>
__global__ void __launch_bounds__(MODE == kCluster ? kBlasCluster : kBlasSingle) k_member_arnoldi(KrylovBufs k) {
  grid_dep_wait();
  __shared__ double red[kRedWords];
  __shared__ double c[34];
  const MemberView mv = member_view(k, blockIdx.y);
  const int len = k.mlen, ldT = k.maxit;
  const int64_t ldv = k.n;
  const int m = k.flags[F_M] + 1;  // the step computed here produces row m of V
  double *vm = k.V + m * ldv + mv.off;
  float *vmf = k.Vf ? k.Vf + m * ldv + mv.off : nullptr;
  const int f = g_first<MODE>(), st = g_stride<MODE>();
  if (mv.flags[F_KSTOP]) {  // uniform over the cluster
    for (int j = f; j < len; j += st) {
      vm[j] = 0.0;
      if (vmf) vmf[j] = 0.0f;
    }
    return;
  }
  const double *Vb = k.V + mv.off;
  const double *v = Vb + (m - 1) * ldv;
  const double *klo = k.klo + mv.off, *kdiag = k.kdiag + mv.off, *kup = k.kup + mv.off;
  double x[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = f + e * st;
    double a = 0.0;
    if (j < len) {
      a = kdiag[j] * v[j];
      if (j > 0) a += klo[j] * v[j - 1];
      if (j + 1 < len) a += kup[j] * v[j + 1];
    }
    x[e] = a;
  }
  __shared__ double cslot[MODE == kCluster ? 3 * kSlot : 1];
  double *const sl2 = MODE == kCluster ? cslot + kSlot : cslot, *const sl3 = MODE == kCluster ? cslot + 2 * kSlot : cslot;
  const bool wr = (MODE == kSingle || blockIdx.x == 0) && (int)threadIdx.x < m;  // writes column m-1 of T
  reg_dots<MODE, E>(len, m, Vb, ldv, x, cslot, 0, red, c);
  const double knorm = sqrt(c[m]);
  const double tq = wr ? c[threadIdx.x] : 0.0;
  reg_axpy<MODE, E>(len, m, Vb, ldv, x, c);
  __syncthreads();  // c is rewritten next
  reg_dots<MODE, E>(len, m, Vb, ldv, x, sl2, 0, red, c);
  if (wr) mv.T[(int64_t)threadIdx.x * ldT + (m - 1)] = tq + c[threadIdx.x];
  reg_axpy<MODE, E>(len, m, Vb, ldv, x, c);
  __syncthreads();
  const double t = sqrt(cgs2_norm2<MODE, E>(m, x, c, sl3, 0, red));
  const bool bd = !(t > 1e-14 * knorm);
  const double it = bd ? 0.0 : 1.0 / t;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = f + e * st;
    if (j < len) {
      const double y = x[e] * it;
      vm[j] = y;
      if (vmf) vmf[j] = (float)y;
    }
  }
  if (g_leader<MODE>()) {
    mv.T[(int64_t)m * ldT + (m - 1)] = bd ? 0.0 : t;
    mv.scal[S_T] = bd ? 0.0 : t;
    mv.scal[S_KNORM] = knorm;
    mv.flags[F_BREAK] = bd ? 1 : 0;
    if (!isfinite(t)) mv.flags[F_NONFIN] = 1;
  }
  cluster_exit<MODE>();
}

// eq. (13) for member blockIdx.y (two CGS passes of its part of z against its basis)
// and its stopping decision; members that had stopped keep their state.
template <int MODE, int E>
__global__ void __launch_bounds__(MODE == kCluster ? kBlasCluster : kBlasSingle) k_member_project(KrylovBufs k, const double *__restrict__ z,
                                                               double tau, KrylovCtl kc, int use_handle,
                                                               cudaGraphConditionalHandle h) {
  grid_dep_wait();
  __shared__ double red[kRedWords];
  __shared__ double c[34];
  const MemberView mv = member_view(k, blockIdx.y);
  const int len = k.mlen;
  const int64_t ldv = k.n;
  if (!mv.flags[F_KSTOP]) {  // the same for every thread of the CTA and the cluster
    __shared__ double cslot[MODE == kCluster ? 3 * kSlot : 1];
    double *const sl2 = MODE == kCluster ? cslot + kSlot : cslot, *const sl3 = MODE == kCluster ? cslot + 2 * kSlot : cslot;
    const int m = mv.flags[F_M] + 1;
    const double *Vb = k.V + mv.off;
    double x[E];
    reg_load<MODE, E>(len, z + mv.off, x);
    reg_dots<MODE, E>(len, m, Vb, ldv, x, cslot, 0, red, c);
    reg_axpy<MODE, E>(len, m, Vb, ldv, x, c);
    __syncthreads();  // c is rewritten next
    reg_dots<MODE, E>(len, m, Vb, ldv, x, sl2, 0, red, c);
    reg_axpy<MODE, E>(len, m, Vb, ldv, x, c);
    __syncthreads();
    const double zz = cgs2_norm2<MODE, E>(m, x, c, sl3, 0, red);
    cluster_exit<MODE>();  // (before the decision changes the flags that the cluster's other CTAs read)
    if (g_leader<MODE>()) {
      mv.scal[S_RES] = mv.flags[F_BREAK] ? 0.0 : fabs(tau * mv.scal[S_T]) * sqrt(zz);
      krylov_decide(mv.scal, mv.flags, kc, 0, h);
    }
  }
  if (last_cta_done(k.counter)) member_totals(k, false, use_handle, h, red);
}

static void member_launch(Ctx &c, const char *fam, double bytes, const void *fn, const KrylovBufs &k, void **args) {
  const int cl = k.cluster > 1 ? k.cluster : 1;
  if (cl > 1) cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (cl > 1) allow_dyn_smem(fn);
  c.launch(fam, bytes, [&] {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)cl, (unsigned)k.members);
    cfg.blockDim = dim3(cl > 1 ? kBlasCluster : kBlasSingle);
    cfg.dynamicSmemBytes = cl > 1 ? kClusterSpreadSmem : 0;
    cfg.stream = c.stream;
    cudaLaunchAttribute attr[2];
    int na = 0;
    if (cl > 1) {
      attr[na].id = cudaLaunchAttributeClusterDimension;
      attr[na].val.clusterDim.x = (unsigned)cl;
      attr[na].val.clusterDim.y = 1;
      attr[na++].val.clusterDim.z = 1;
    }
    if (c.pdl) {
      attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[na++].val.programmaticStreamSerializationAllowed = 1;
    }
    cfg.attrs = attr;
    cfg.numAttrs = na;
    cudaLaunchKernelExC(&cfg, fn, args);
  });
}

#define PD_MEMBER_E(E, KERNEL, MODE)                                                                 \
  ((E) <= 1 ? (const void *)KERNEL<MODE, 1>                                                         \
            : (E) == 2 ? (const void *)KERNEL<MODE, 2>                                              \
                       : (E) == 4 ? (const void *)KERNEL<MODE, 4>                                   \
                                  : (E) == 8 ? (const void *)KERNEL<MODE, 8> : (const void *)KERNEL<MODE, 16>)
#define PD_MEMBER_BY_E(K, KERNEL)                                                                    \
  ((K).cluster > 1 ? PD_MEMBER_E(reg_elems((K).mlen, (K).cluster * kBlasCluster), KERNEL, kCluster) \
                   : PD_MEMBER_E(reg_elems((K).mlen, kBlasSingle), KERNEL, kSingle))

// Clusters of 8 CTAs, of 4 while those of all members would not fit the SMs side by side; 0: one CTA
// per member (more members than clusters of 4 leave room for, or short problems).  Eight clusters of 16
// were slower than one CTA each (8 x 2048 rows: 16.3 / 21.8 / 22.4 us).  A caller's size (want > 0) is taken
// as it is, as for single problems; clusters that do not fit side by side run one after another.
int member_cluster_size(int members, int len, int want) {
  if (want <= 0) {
    want = 8;
    while (want >= 4 && want * members > sm_count()) want >>= 1;
  }
  return want < 4 || len < 256 ? 0 : krylov_cluster_size(want);
}

void launch_member_init(Ctx &c, KrylovBufs &k, const double *b, int use_handle, cudaGraphConditionalHandle h) {
  void *args[] = {&k, (void *)&b, &use_handle, &h};
  member_launch(c, "krylov_init", (double)k.n * 16, PD_MEMBER_BY_E(k, k_member_init),
                k, args);
}

void launch_member_arnoldi(Ctx &c, KrylovBufs &k) {
  void *args[] = {&k};
  member_launch(c, "krylov_arnoldi", (double)k.n * 8.0 * 8,
                PD_MEMBER_BY_E(k, k_member_arnoldi), k, args);
}

void launch_member_project(Ctx &c, KrylovBufs &k, const double *z, double tau, const KrylovCtl &kc0, int use_handle,
                           cudaGraphConditionalHandle h) {
  KrylovCtl kc = kc0;
  void *args[] = {&k, (void *)&z, &tau, &kc, &use_handle, &h};
  member_launch(c, "krylov_project", (double)k.n * 8.0 * 6,
                PD_MEMBER_BY_E(k, k_member_project), k, args);
}

}  // namespace pd
