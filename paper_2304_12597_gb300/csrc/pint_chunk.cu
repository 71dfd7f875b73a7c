// The binary32 parallel-in-time loop with chunks in registers: the shifted solves
// ((1 - pi_k) I + tau K) y_k = r_k of pint.cu for plans that neither store factors nor run the
// FP64 zero-frequency lane nor have rows far from diagonal dominance (those keep k_pint).
//
// One team of P lanes solves one tridiagonal block of blen <= P M rows; lane t owns the M
// consecutive rows from t M in registers.
//  1. Forward: rows 0..M-2 of the chunk become x_i + aa_i X + cc_i x_{i+1} = r_i, where X is the
//     last unknown of the chunk before; beside it, x_0 = D - A X + w L with the chunk's own last
//     unknown L.
//  2. Row M-1 and the next chunk's x_0 give one row in (X, L, next L) per chunk: P rows, solved by
//     parallel cyclic reduction on unit-diagonal rows (P <= 32: shuffles; wider teams: shared memory).
//  3. Back substitution from L: x_i = r_i - aa_i X - cc_i x_{i+1}.
// Elimination is without pivoting inside principal blocks, as in pint.cu.
//
// Every row carries its excess, the sum of its coefficients, instead of its diagonal: a pivot is
// then excess - (off-diagonals), and the excess itself is updated by row operations of its own.
// For M-matrices (heat, upwinding: off-diagonals <= 0, excess >= 0) all these are sums of terms
// of one sign (with a complex shift: terms within a quarter plane), so pivots lose nothing to
// cancellation, however ill-conditioned the small shifts make the system (A. K. Alfa, J. Xue,
// Q. Ye, Math. Comp. 71 (2002): elimination of diagonally dominant M-matrices from their
// off-diagonals and row sums).  With the diagonal instead, 1 - lo up / pivot cancels to the
// row's small excess and a binary32 solve of the low frequencies is off by kappa u: 2e-4 on
// 1023 x 1024 heat, against 1e-5 this way, and the sum tau (lo + diag + up) no longer depends on
// the rounding of the three coefficients to binary32.  The refinement then contracts by 1e-5 to
// 1e-6 a sweep instead of 1e-3 to 1e-4, at about 25 % more arithmetic in this kernel (2D: 43 -> 44 us
// per loop): advdiff1d_4095x2048 and heat2d_255x255x256 take 3 solves instead of 4 (1530 ->
// 1160 us, 2964 -> 2234 us), 32 x heat1d_1023x1024 takes 3 instead of 5 (5336 -> 3297 us).
// For other signs the same identities hold, with the rounding of the off-diagonals in place of the
// diagonal's: harmless in rows that are dominant or nearly so, the only ones that come here
// (suits_excess in plan.cu; a graded symmetric operator with off-diagonals 600 times the diagonal
// left the refinement short of convergence).
//
// What bounds it: latency.  A lane walks a serial chain of 16 pivots, and at 168 registers an SM
// holds 12 warps (14 % of its slots), which issue in 49 % of the cycles (255 x 255 x 256); wide teams
// (blocks of more than 512 rows; 16 warps, 42 % at 4095 x 2048) also wait at a barrier per PCR level
// and, in one CTA of 256, for each frequency's loads.  105 thread instructions per row at 255 rows a
// block, 156 at 4095.  Against k_pint's two separators per chunk
// of 8 rows held in shared memory (230 instructions per row) this takes 16 rows per lane (half the PCR
// levels per row), keeps aa, cc, r in registers, moves tau K as one 16-byte shared load per row, and,
// up to teams of 128 lanes, prefetches the next frequency's right-hand side with cp.async while this
// one is solved.
// Measured per launch (one GB300, k_pint -> this kernel; b pass / h_k pass):
//   2D 255 blocks of 255 rows, 129 frequencies     94 / 98 us   -> 45 / 41 us
//   2D 127 blocks of 127 rows, 257 frequencies     67 / 71 us   -> 24 / 22 us
//   32 blocks of 1023 rows, 513 frequencies       204 / 236 us  -> 85 / 92 us
//   one block of 4095 rows, 1025 frequencies       65 / 67 us   -> 38 / 36 us
//   one block of 511 rows, 17 frequencies         12.9 / 13.8 us -> 9.7 / 7.9 us (latency)
#include <algorithm>

#include "pd_internal.h"

namespace pd {

namespace {

__device__ __forceinline__ void cp_async8(void *smem, const void *g) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(s), "l"(g));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

using C = cpx<float>;
// -a b
__device__ __forceinline__ C nmul(C a, C b) {
  return mk<float>(fmaf(a.y, b.y, -(a.x * b.x)), -fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ C sub1(C a, float s) { return mk<float>(a.x - s, a.y); }
__device__ __forceinline__ C shfl_up(C v, int d, int w) {
  return mk<float>(__shfl_up_sync(0xffffffffu, v.x, d, w), __shfl_up_sync(0xffffffffu, v.y, d, w));
}
__device__ __forceinline__ C shfl_dn(C v, int d, int w) {
  return mk<float>(__shfl_down_sync(0xffffffffu, v.x, d, w), __shfl_down_sync(0xffffffffu, v.y, d, w));
}

__device__ __forceinline__ C fma_c(C a, C b, C c) {  // a + b c
  return mk<float>(fmaf(-b.y, c.y, fmaf(b.x, c.x, a.x)), fmaf(b.y, c.x, fmaf(b.x, c.y, a.y)));
}

// A unit-diagonal row a x_lo + x + c x_hi = d with its excess g = 1 + a + c carried beside it.
struct SepRow {
  C a, c, d, g;
};
// One PCR level, given the neighbours' rows.  A row without a lower (upper) neighbour has a = 0
// (c = 0), so whatever finite row stands in for the missing neighbour drops out.
__device__ __forceinline__ void pcr_level(SepRow &r, const SepRow &l, const SepRow &h, bool last) {
  const C a = nmul(r.a, l.a), c = nmul(r.c, h.c);
  const C g = fnms(fnms(r.g, r.a, l.g), r.c, h.g);
  const C q = recip(sub(sub(g, a), c));
  r.d = mul(fnms(fnms(r.d, r.a, l.d), r.c, h.d), q);
  if (!last) {
    r.a = mul(a, q);
    r.c = mul(c, q);
    r.g = mul(g, q);
  }
}

}  // namespace

// What a launch does besides solving (compile-time, so that each keeps only its registers).
enum ChunkMode { kPlain = 0, kAcc = 1, kDots = 2 };

// PW: lanes per team (8, 16 or 32, several teams per CTA), or 0 for one team of blockDim.x
// lanes.  TS: complex values per team buffer, P (M + 1): one pad slot per chunk, so that the
// lanes' chunk accesses and the row-wise copies are both free of bank conflicts.
template <int M, int PW, int MODE, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_pint_chunk(PintGeom g, PintArgs<float> a) {
  grid_dep_wait();
  if (a.skip_flag && *a.skip_flag) return;
  if (a.skip_flag2 && *a.skip_flag2) return;
  const int P = PW ? PW : (int)blockDim.x;
  const int teams = PW ? (int)blockDim.x / PW : 1;
  const int TS = P * (M + 1);
  const int t = PW ? (int)threadIdx.x % PW : (int)threadIdx.x;   // lane of the team
  const int team = PW ? (int)threadIdx.x / PW : 0;               // team of the CTA
  const int blk = (int)blockIdx.x / g.R, rr = (int)blockIdx.x - blk * g.R;
  const int blen = g.blen;
  const int64_t off = (int64_t)blk * blen;

  extern __shared__ __align__(16) unsigned char smraw[];
  float4 *cs = reinterpret_cast<float4 *>(smraw);                // tau lo, tau (lo + diag + up), tau up, vector
  constexpr int NB = NT >= 256 ? 1 : 2;                          // right-hand-side buffers
  C *bufs = reinterpret_cast<C *>(cs + TS);                      // [NB][teams][TS]
  double2 *red = reinterpret_cast<double2 *>(bufs + (size_t)NB * teams * TS);  // PW == 0: [warps][mdots]

  const bool has_r = a.R != nullptr;
  // the vector of the block's rows: subtracted from every R[k], or the right-hand side itself
  const float *rvec = a.rvec;
  int mdots = MODE == kDots ? a.mdots : 0;
  if (a.mcount) {
    const int m = *a.mcount + 1;
    rvec = a.V + (int64_t)m * a.ldv;
    if (MODE == kDots) mdots = m;
  }
  // frequencies of this CTA's pass `it`: team q of it solves k = (it R + rr) teams + q
  const int kstep = g.R * teams;
  const int kfirst = rr * teams;

  // Row-wise view of the CTA's (or, PW > 0, the warp's) team buffers: copy j of a thread moves
  // element lin = j stride + thread, i.e. row element e of team q, so that a warp moves 256
  // contiguous bytes where a block has them.
  constexpr int WT = PW ? 32 / PW : 1;           // teams per warp
  constexpr int RL = PW ? PW * M : 0;            // padded row length of a team
  const int lane = (int)threadIdx.x & 31;
  const int wteam = PW ? ((int)threadIdx.x >> 5) * WT : 0;
  auto sync_team = [&]() {
    if constexpr (PW != 0)
      __syncwarp();
    else
      __syncthreads();
  };
  auto load_rows = [&](int b, int kb) {  // R rows of frequencies kb (+ team) into buffer b
#pragma unroll
    for (int j = 0; j < M; ++j) {
      int q, e;
      if constexpr (PW != 0) {
        const int lin = j * 32 + lane;
        q = wteam + lin / RL;
        e = lin % RL;
      } else {
        q = 0;
        e = t + j * P;
      }
      C *dst = bufs + ((size_t)b * teams + q) * TS + e + e / M;
      const int k = kb + q;
      if (e < blen && k < g.nf)
        cp_async8(dst, a.R + (int64_t)k * a.ldr + off + e);
      else
        *dst = mk<float>(0.0f, 0.0f);
    }
  };

  if (NB == 2 && has_r && kfirst < g.nf) load_rows(0, kfirst);
  cp_async_commit();

  // stage tau K and the vector once per CTA (its block does not change): SB rows per thread and
  // round, their loads all issued before any is used (one memory latency per round and basis row)
  {
    constexpr int SB = 8;
    const int m = a.xm_count ? *a.xm_count : 0;
    const double *xy = a.xm_count ? a.xm_y + (int64_t)(blk / (a.xm_bpm > 1 ? a.xm_bpm : 1)) * a.xm_ldy : nullptr;
    const int n = P * M, nt = (int)blockDim.x;
    for (int e0 = threadIdx.x; e0 < n; e0 += SB * nt) {
      float4 q[SB];
#pragma unroll
      for (int u = 0; u < SB; ++u) {
        const int e = e0 + u * nt;
        const bool in = e < blen;
        // rows outside the block do not exist: its first lo and last up are zero
        q[u].x = in && e > 0 ? a.tlo[off + e] : 0.0f;
        q[u].y = in ? a.texc[off + e] : 1.0f;
        q[u].z = in && e + 1 < blen ? a.tup[off + e] : 0.0f;
        q[u].w = in && rvec && !xy ? rvec[off + e] : 0.0f;
      }
      if (xy) {  // x_m = V_m y_m (Algorithm 3 weights it by alpha^{1/l})
        for (int i = 0; i < m; ++i) {
          const float yi = (float)xy[i];
          const float *vi = a.V + (int64_t)i * a.ldv + off;
#pragma unroll
          for (int u = 0; u < SB; ++u) q[u].w += yi * (e0 + u * nt < blen ? vi[e0 + u * nt] : 0.0f);
        }
#pragma unroll
        for (int u = 0; u < SB; ++u) q[u].w *= (float)a.xm_scale;
        if (rr == 0 && a.xm_out) {
          double vd[SB];
#pragma unroll
          for (int u = 0; u < SB; ++u) vd[u] = 0.0;
          for (int i = 0; i < m; ++i) {
            const double *vi = a.xm_Vd + (int64_t)i * a.ldv + off;
#pragma unroll
            for (int u = 0; u < SB; ++u) vd[u] += xy[i] * (e0 + u * nt < blen ? vi[e0 + u * nt] : 0.0);
          }
#pragma unroll
          for (int u = 0; u < SB; ++u)
            if (e0 + u * nt < blen) a.xm_out[off + e0 + u * nt] = vd[u];
        }
      }
#pragma unroll
      for (int u = 0; u < SB; ++u) {
        const int e = e0 + u * nt;
        if (e < n) cs[e + e / M] = q[u];
      }
    }
  }
  __syncthreads();

  float acc[M];
  if (MODE == kAcc) {
#pragma unroll
    for (int i = 0; i < M; ++i) acc[i] = 0.0f;
  }
  const float4 *mc = cs + t * (M + 1);
  const bool tail = t * M + M > blen;  // the chunk holds rows past the block's end

  int b = 0;
  for (int kb = kfirst; kb < g.nf; kb += kstep, b ^= NB - 1) {
    const int k = kb + team;
    const bool live = k < g.nf;
    C *buf = bufs + ((size_t)b * teams + team) * TS;
    if (has_r) {
      if (NB == 1)
        load_rows(0, kb);
      else if (kb + kstep < g.nf)
        load_rows(b ^ 1, kb + kstep);
      cp_async_commit();
      cp_async_wait<NB - 1>();
      sync_team();
    }
    const C s = a.shift_t[live ? k : 0];
    C *my = buf + t * (M + 1);

    // 1. forward: row i as (aa, 1, cc), its excess gg, and x_0 = D - A X + w x_{i+1} with the
    // excess gm = 1 + A - w
    C aa[M], cc[M], r[M];
    C D, A, w, gm, gg, sep_a, sep_g, sep_d;
    float sep_up;
#pragma unroll
    for (int i = 0; i < M; ++i) {
      const float4 q = mc[i];
      C ri = has_r ? my[i] : mk<float>(q.w, 0.0f);
      if (has_r) ri.x -= q.w;
      // rows past the block's end: 1 x = 0, whatever the shift
      const C e = (tail && t * M + i >= blen) ? mk<float>(1.0f, 0.0f) : mk<float>(s.x + q.y, s.y);
      const C al = i == 0 ? mk<float>(q.x, 0.0f) : scal(-q.x, aa[i - 1]);
      const C g1 = i == 0 ? e : fnms_r(e, q.x, gg);
      if (i > 0) ri = fnms_r(ri, q.x, r[i - 1]);
      if (i < M - 1) {
        const C rd = recip(sub1(sub(g1, al), q.z));
        aa[i] = i == 0 ? scal(q.x, rd) : mul(al, rd);
        cc[i] = scal(q.z, rd);
        gg = mul(g1, rd);
        r[i] = mul(ri, rd);
        D = i == 0 ? r[0] : fma_c(D, w, r[i]);
        A = i == 0 ? aa[0] : fma_c(A, w, aa[i]);
        gm = i == 0 ? gg : fma_c(gm, w, gg);
        w = i == 0 ? scal(-1.0f, cc[0]) : nmul(w, cc[i]);
      } else {
        sep_a = al;
        sep_g = g1;
        sep_d = ri;
        sep_up = q.z;
      }
    }
    // 2. one row per chunk in (X, L, next L), unit diagonal, and its PCR
    auto sep_row = [&](C An, C wn, C gn, C Dn) {
      SepRow v;
      v.a = sep_a;
      v.c = scal(sep_up, wn);
      v.g = fnms_r(sep_g, sep_up, gn);
      const C q = recip(sub(sub(v.g, v.a), v.c));
      v.a = mul(v.a, q);
      v.c = mul(v.c, q);
      v.g = mul(v.g, q);
      v.d = mul(fnms_r(sep_d, sep_up, Dn), q);
      return v;
    };
    C L, X;
    if constexpr (PW != 0) {
      SepRow v = sep_row(A, shfl_dn(w, 1, PW), shfl_dn(gm, 1, PW), shfl_dn(D, 1, PW));
#pragma unroll
      for (int sg = 1; sg < PW; sg <<= 1) {
        const SepRow lo{shfl_up(v.a, sg, PW), shfl_up(v.c, sg, PW), shfl_up(v.d, sg, PW), shfl_up(v.g, sg, PW)};
        const SepRow hi{shfl_dn(v.a, sg, PW), shfl_dn(v.c, sg, PW), shfl_dn(v.d, sg, PW), shfl_dn(v.g, sg, PW)};
        pcr_level(v, lo, hi, 2 * sg >= PW);
      }
      L = v.d;
      X = shfl_up(L, 1, PW);
      if (t == 0) X = mk<float>(0.0f, 0.0f);
    } else {
      // the exchanged rows sit in the lanes' own chunk slots of the buffer, which each lane has
      // read by now: eight slots of a lane, in two sets of four that alternate.  A set is
      // rewritten two levels later, past the barrier that every lane reaches after reading it.
      my[0] = D;
      my[1] = w;
      my[2] = gm;
      __syncthreads();
      const C *nx = my + (t + 1 < P ? M + 1 : 0);
      SepRow v = sep_row(A, nx[1], nx[2], nx[0]);
      int lv = 4;
      for (int sg = 1; sg < P; sg <<= 1, lv ^= 4) {
        C *own = my + lv;
        own[0] = v.a;
        own[1] = v.c;
        own[2] = v.d;
        own[3] = v.g;
        __syncthreads();
        const C *lo = own - (t >= sg ? sg * (M + 1) : 0), *hi = own + (t + sg < P ? sg * (M + 1) : 0);
        pcr_level(v, SepRow{lo[0], lo[1], lo[2], lo[3]}, SepRow{hi[0], hi[1], hi[2], hi[3]}, 2 * sg >= P);
      }
      L = v.d;
      my[lv] = L;
      __syncthreads();
      X = t > 0 ? my[lv - (M + 1)] : mk<float>(0.0f, 0.0f);
      __syncthreads();  // x goes into the slots next
    }

    // 3. back substitution, and the accumulation of b (eq. 7)
    float ox = 0.0f, oy = 0.0f;
    if (MODE == kAcc && live) {
      if (a.omega_t) {
        ox = a.omega_t[k].x;
        oy = a.omega_t[k].y;
      } else {
        ox = (float)a.omega[k].x;
        oy = (float)a.omega[k].y;
      }
    }
    C x = L;
    const bool out = a.Y != nullptr || MODE == kDots;
#pragma unroll
    for (int i = M - 1; i >= 0; --i) {
      if (i < M - 1) x = fnms(fnms(r[i], aa[i], X), cc[i], x);
      if (MODE == kAcc) acc[i] += ox * x.x - oy * x.y;
      if (out) my[i] = x;
    }
    if (out) sync_team();

    // 4. store
    if (a.Y) {
#pragma unroll
      for (int j = 0; j < M; ++j) {
        int q, e;
        if constexpr (PW != 0) {
          const int lin = j * 32 + lane;
          q = wteam + lin / RL;
          e = lin % RL;
        } else {
          q = 0;
          e = t + j * P;
        }
        if (e < blen && kb + q < g.nf)
          a.Y[(int64_t)(kb + q) * a.ldy + off + e] = bufs[((size_t)b * teams + q) * TS + e + e / M];
      }
    }
    // 5. g_k = V_m^T y_k: sums over a warp in binary32, over a team's warps in FP64
    if (MODE == kDots && mdots > 0) {
      C yv[M];
#pragma unroll
      for (int j = 0; j < M; ++j) {
        const int e = t + j * P;
        yv[j] = e < blen ? buf[e + e / M] : mk<float>(0.0f, 0.0f);
      }
      for (int q = 0; q < mdots; ++q) {
        const float *vq = a.V + (int64_t)q * a.ldv + off;
        float sx = 0.0f, sy = 0.0f;
#pragma unroll
        for (int j = 0; j < M; ++j) {
          const int e = t + j * P;
          const float v = e < blen ? vq[e] : 0.0f;
          sx += v * yv[j].x;
          sy += v * yv[j].y;
        }
#pragma unroll
        for (int o = (PW ? PW : 32) / 2; o > 0; o >>= 1) {
          sx += shfl_xor(sx, o);
          sy += shfl_xor(sy, o);
        }
        if constexpr (PW != 0) {
          if (t == 0 && live) a.gpart[((int64_t)k * g.nblk + blk) * mdots + q] = make_double2((double)sx, (double)sy);
        } else {
          if (lane == 0) red[(threadIdx.x >> 5) * mdots + q] = make_double2((double)sx, (double)sy);
        }
      }
      if constexpr (PW == 0) {
        __syncthreads();
        for (int q = t; q < mdots; q += P) {
          double sx = 0.0, sy = 0.0;
          for (int w = 0; w < (P >> 5); ++w) {
            sx += red[w * mdots + q].x;
            sy += red[w * mdots + q].y;
          }
          a.gpart[((int64_t)k * g.nblk + blk) * mdots + q] = make_double2(sx, sy);
        }
      }
    }
    // the next pass writes this buffer
    sync_team();
  }

  if (MODE == kAcc) {
    // the CTA's partial row of b: its teams' sums added in FP64 in a fixed order
    cp_async_wait<0>();
    __syncthreads();
    float *fb = reinterpret_cast<float *>(bufs);
#pragma unroll
    for (int i = 0; i < M; ++i) fb[(size_t)team * TS + t * (M + 1) + i] = acc[i];
    __syncthreads();
    for (int e = threadIdx.x; e < blen; e += blockDim.x) {
      double sum = 0.0;
      for (int q = 0; q < teams; ++q) sum += (double)fb[(size_t)q * TS + e + e / M];
      a.acc_part[((int64_t)blk * g.R + rr) * blen + e] = sum;
    }
  }
}

// Rows per lane and lanes per team.  Sixteen rows per lane from 65 rows on (fewest PCR levels
// per row that fit the register budget); blocks of up to 64 rows take eight, so that their
// teams still fill a warp with four blocks.
PintGeom pint_chunk_geometry(int nf, int nblk, int blen) {
  PintGeom g{};
  g.chunk = 1;
  g.nf = nf;
  g.nblk = nblk;
  g.blen = blen;
  g.M = blen <= 64 ? 8 : 16;
  int P = 8;
  while (P * g.M < blen) P <<= 1;
  g.P = P;
  const int nt = std::max(P, 64);
  g.teams_per_cta = P <= 32 ? nt / P : 1;
  // Splits of the frequency range: the fewest passes over the resident CTAs (384 threads per
  // SM by registers), a pass being one frequency per team plus a start-up worth one.
  const int64_t slots = (int64_t)sm_count() * (g.M == 8 ? 8 : P >= 256 ? 2 : 384 / nt);
  const int rmax = (nf + g.teams_per_cta - 1) / g.teams_per_cta;
  int64_t best = -1;
  g.R = 1;
  for (int R = 1; R <= rmax; ++R) {
    const int64_t waves = ((int64_t)nblk * R + slots - 1) / slots;
    const int64_t iters = (rmax + R - 1) / R;
    const int64_t cost = waves * (iters + 1);
    if (best < 0 || cost < best) {
      best = cost;
      g.R = R;
    }
  }
  g.acc_rows = g.R;
  return g;
}

template <int M, int PW, int NT, int MINB>
static void chunk_launch(Ctx &c, const PintGeom &g, const PintArgs<float> &a) {
  const bool dots = a.mcount ? a.want_dots != 0 : (a.V && a.mdots > 0);
  const int mode = dots ? kDots : (a.omega ? kAcc : kPlain);
  const int threads = PW ? std::max(g.P, 64) : g.P;
  const int teams = g.teams_per_cta;
  const size_t TS = (size_t)g.P * (M + 1);
  const int md = a.mcount ? a.mdots_max : a.mdots;
  const size_t smem = TS * sizeof(float4) + (NT >= 256 ? 1 : 2) * teams * TS * sizeof(C) +
                      (PW || !dots ? 0 : (size_t)(g.P / 32) * md * sizeof(double2));
  double bytes = 0.0;
  const double per = (double)g.nf * g.nblk * g.blen;
  if (a.R) bytes += per * sizeof(C);
  if (a.Y) bytes += per * sizeof(C);
  const char *fam = mode == kDots ? "pint_dots_f32" : (mode == kAcc ? "pint_acc_f32" : "pint_store_f32");
  c.launch(fam, bytes, [&] {
    auto kern = mode == kDots ? k_pint_chunk<M, PW, kDots, NT, MINB>
                              : (mode == kAcc ? k_pint_chunk<M, PW, kAcc, NT, MINB> : k_pint_chunk<M, PW, kPlain, NT, MINB>);
    if (smem > 48 * 1024) allow_dyn_smem((const void *)kern);
    pdl_launch(c.pdl, kern, dim3((unsigned)(g.nblk * g.R)), dim3(threads), smem, c.stream, g, a);
  });
}

void launch_pint_chunk(Ctx &c, const PintGeom &g, const PintArgs<float> &a) {
  if (g.M == 8)
    chunk_launch<8, 8, 64, 8>(c, g, a);
  else if (g.P == 8)
    chunk_launch<16, 8, 64, 6>(c, g, a);
  else if (g.P == 16)
    chunk_launch<16, 16, 64, 6>(c, g, a);
  else if (g.P == 32)
    chunk_launch<16, 32, 64, 6>(c, g, a);
  else if (g.P == 64)
    chunk_launch<16, 0, 64, 6>(c, g, a);
  else if (g.P == 128)
    chunk_launch<16, 0, 128, 3>(c, g, a);
  else
    chunk_launch<16, 0, 256, 2>(c, g, a);
}

}  // namespace pd
