// jacobi.cu - FP64 symmetric eigensolver for the HOSVD Gram matrices (Fig. 1B) and the
// choice of the truncating isometry.
//
// jacobi_kernel: one CTA per matrix. Cyclic two-sided Jacobi in round-robin (tournament)
// order: each round rotates n/2 disjoint index pairs at once, so every 2x2 block of A is
// updated by exactly one thread and the rounds need only block barriers. The tournament runs
// separately inside each connected component of A's nonzero pattern (exact zeros between
// components stay exact zeros), which quarters the work when the Gram matrix splits by Z2
// charge. A pair is
// rotated when |a_pq| > max(1e-18 ||G||_F, 2^-52 sqrt|a_pp a_qq|); a sweep after which no pair
// passes that test ends the loop, and max_sweeps sweeps (kJacobiMaxSweeps unless the context
// overrides it) raise the no-convergence status
// (results are still written). Then: eigenvalues sorted descending, the discarded sum
// eps = sum_{j >= chi} lambda_j, and the first chi eigenvectors in the canonical gauge:
// eigenvalues closer than cluster_tau * lambda_0 form a cluster (cluster_tau is set
// above the rounding noise of the Gram matrix: 1e-10 when the tensors are FP64, 1e-6
// when they are stored in FP32); inside a cluster the
// basis is built by repeatedly taking the unit vector e_i with the longest projection on
// the not-yet-covered part of the cluster's eigenspace (lowest i within a relative
// tie_rel of the longest: 1e-8 for FP64 tensors, 1e-4 for FP32-stored ones, whose noise
// would otherwise break exact symmetric ties at random) and normalising that projection. This gauge depends only on the
// eigenspaces, so it does not depend on the eigensolver.
//
// The FP64 pipe bounds it (measured: one warp issues an FP64 instruction every 64 cycles, whatever its lanes or
// dependences, an SM one every 19), so a round costs 64 cycles per FP64 instruction of its longest chain, or 19
// per warp instruction of its blocks, and even comparisons and conversions count. So: A is kept as its upper triangle, 13 FP64 instructions per 2x2 block off
// the diagonal; the rotation's tangent is computed in FP32 (from the bits) and its cosine refined to FP64 from an
// FP32 start, 7 FP64 instructions; thresholds, sorting and tests are integer operations on the bits; a round in
// which nothing rotates is skipped; and the eigenvector matrix is not accumulated: the rotations are logged, and
// the columns that are needed (the clusters that reach into the first chi; 8 of 64 at D = 8) are formed at the
// end by applying the log backwards to unit vectors, one column per group of lanes without block barriers.
//
// select_kernel: per transverse direction, the side (nu or nu') with the smaller
// discarded sum (a difference within side_rel (eps + eps') + 1e-13 lambda_0 is a tie and
// goes to nu; side_rel = 1e-9 for FP64 tensors, 1e-6 for FP32 ones), then modified Gram-Schmidt in FP64 on the kept vectors, and copies of U in
// FP64 and in the storage precision.
#include <math.h>

#include "common.cuh"

namespace hotrg {

constexpr int kJT = 544;            // most threads of a Jacobi CTA: the 496 + 32 blocks of n = 64 in one pass

// Local indices of pair i of round r among m (even) players; r < m - 1, i < m / 2.
__device__ __forceinline__ void rr_pair(int r, int i, int m, int& p, int& q) {
  if (i == 0) {
    p = r;
    q = m - 1;
  } else {
    p = r + i;
    if (p >= m - 1) p -= m - 1;
    q = r - i;
    if (q < 0) q += m - 1;
  }
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
}

// e-th entry (row-major) of the upper triangle, diagonal included, of an h x h grid.
__device__ __forceinline__ void tri_index(int e, int h, int& P, int& Q) {
  // rows start at s(P) = P h - P (P - 1) / 2; invert with a float square root, then fix up
  const float b = 2.0f * h + 1.0f;
  int r = (int)((b - sqrtf(b * b - 8.0f * (float)e)) * 0.5f);
  r = r < 0 ? 0 : (r > h - 1 ? h - 1 : r);
  while (r > 0 && r * h - r * (r - 1) / 2 > e) --r;
  while (r + 1 < h && (r + 1) * h - (r + 1) * r / 2 <= e) ++r;
  P = r;
  Q = r + (e - (r * h - r * (r - 1) / 2));
}

// Place of entry (i, j) in the packed upper triangle of an n x n matrix.
__device__ __forceinline__ int packed(int i, int j, int n) {
  const int lo = min(i, j), hi = max(i, j);
  return lo * (2 * n - 1 - lo) / 2 + hi;
}

// v 2^-(em - 1023) as a float (toward zero; 0 below FP32's range), and a normal or zero float as a double: by
// their bits, without the FP64 pipe. em: biased exponent not below v's.
__device__ __forceinline__ float scaled_float(double v, int em) {
  const int hi = __double2hiint(v), e = ((hi >> 20) & 0x7ff) - em + 127;
  const uint32_t m = ((uint32_t)hi & 0xfffffu) << 3 | (uint32_t)__double2loint(v) >> 29;
  return __int_as_float(e <= 0 ? 0 : (int)((uint32_t)hi & 0x80000000u | (uint32_t)e << 23 | m));
}
__device__ __forceinline__ double widen(float f) {
  const uint32_t b = __float_as_uint(f);
  const uint32_t hi = (b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + (896u << 20));
  return (b & 0x7f800000u) ? __hiloint2double((int)hi, (int)(b << 29)) : 0.0;
}

__global__ void __launch_bounds__(kJT) jacobi_kernel(const __grid_constant__ EigPack jobs, int njobs, int use_smem,
                                                     int region, double cluster_tau, double tie_rel, int max_sweeps,
                                                     int* status) {
  extern __shared__ double dyn[];          // region doubles (A, later the columns in progress), then the block list
  // one slot per rotation pair of a round: at most n (ceil(m_c / 2) <= m_c per component)
  __shared__ double2 ct[kMaxGramN];        // cosine and tangent
  __shared__ short2 pq[kMaxGramN];         // the pair's indices (second: -1 where the component is odd)
  __shared__ double lam[kMaxGramN];
  __shared__ long long key[kMaxGramN];
  __shared__ double nrmv[kMaxGramN];
  __shared__ int perm[kMaxGramN], cstart[kMaxGramN + 1];
  __shared__ int ired[kJT / 32];
  __shared__ float fred[kJT / 32];
  __shared__ int comp[kMaxGramN];          // component label: its smallest index
  __shared__ int cnum[kMaxGramN];          // component number of an index
  __shared__ int mem[kMaxGramN];           // indices grouped by component
  __shared__ int cbeg[kMaxGramN + 1];      // component c: mem[cbeg[c] .. cbeg[c + 1])
  __shared__ int poff[kMaxGramN + 1];      // first pair slot of component c
  __shared__ int toff[kMaxGramN + 1];      // first 2x2 block of component c
  __shared__ int sz[kMaxGramN];
  __shared__ int ncomp, rmax, npmax, ncl;

  // job blockIdx.x % njobs of batch element blockIdx.x / njobs
  const int64_t bidx = blockIdx.x / njobs;
  EigJob jb = jobs.j[blockIdx.x - bidx * njobs];
  jb.G += bidx * jobs.sG;
  jb.work += bidx * jobs.sWork;
  jb.lam += bidx * jobs.sLam;
  jb.U += bidx * jobs.sU;
  jb.eps += bidx * jobs.sEps;
  jb.degenerate += bidx * jobs.sDeg;
  const int n = jb.n, chi = jb.chi;
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31;
  double* W = jb.work;                     // [column][n]: the needed eigenvectors
  double* V = W + (int64_t)n * n;          // [n][n], rows
  double* Aw = V + (int64_t)n * n;
  double2* log = (double2*)(Aw + (use_smem ? 0 : packed_doubles(n)));
  short2* logi = (short2*)(log + (int64_t)jobs.log_sweeps * n * n);
  double* A = use_smem ? dyn : Aw;         // use_smem: every job of the launch has n <= kJacobiSmemN
  uint32_t* blk = (uint32_t*)(dyn + region);

  // the upper triangle of G (the merged Gram is symmetric up to summation order), scaled by a power
  // of two to a largest magnitude in [1, 2), so that squares neither overflow nor vanish
  int big = 0;                             // exponent bits of the largest magnitude
  for (int e = tid; e < n * n; e += nthr) {
    const int i = e / n, j = e - i * n;
    if (i <= j) big = max(big, __double2hiint(jb.G[e]) & 0x7ff00000);
  }
  big = __reduce_max_sync(0xffffffffu, big);
  if (lane == 0) ired[tid >> 5] = big;
  __syncthreads();
  big = 0;
  for (int w = 0; w < nthr >> 5; ++w) big = max(big, ired[w]);
  // 2^-e and 2^e; no scaling of zeros, infinities, NaN and magnitudes near the ends of the range
  if (big < (24 << 20) || big > (2022 << 20)) big = 1023 << 20;
  const double up = __hiloint2double(0x7fe00000 - big, 0), down = __hiloint2double(big, 0);
  float fro = 0;
  for (int e = tid; e < n * n; e += nthr) {
    const int i = e / n, j = e - i * n;
    if (i > j) continue;
    const double g = jb.G[e] * up;
    A[packed(i, j, n)] = g;
    const float f = (float)g;
    fro = fmaf(i == j ? f : 2 * f, f, fro);
  }
  for (int off = 16; off > 0; off >>= 1) fro += __shfl_xor_sync(0xffffffffu, fro, off);
  if (lane == 0) fred[tid >> 5] = fro;
  __syncthreads();
  fro = 0;
  for (int w = 0; w < nthr >> 5; ++w) fro += fred[w];
  // Exponent of 1e-18 ||G||_F, and the test of a pair by exponents: true for every |a_pq| above
  // max(1e-18 ||G||_F, 2^-52 sqrt|a_pp a_qq|), and for some down to a quarter of it.
  const int e_abs = (__double2hiint(1e-18 * (double)sqrtf(fro)) >> 20) & 0x7ff;
  auto rotates = [&](double apq, double app, double aqq) {
    const int e = (__double2hiint(apq) >> 20) & 0x7ff;
    const int ep = (__double2hiint(app) >> 20) & 0x7ff, eq = (__double2hiint(aqq) >> 20) & 0x7ff;
    return e >= e_abs && e != 0 && e != 0x7ff && 2 * e + 2 > ep + eq - 104;
  };
  auto nonzero = [](double v) { return ((unsigned long long)__double_as_longlong(v) << 1) != 0ull; };

  // ---- connected components of the nonzero pattern of A. A rotation of a pair inside one
  // component leaves the entries between components exactly zero, so each component is
  // diagonalised by its own round-robin tournament and the rest is skipped, exactly. With h = 0
  // the Gram matrices of the Ising tensors split this way by the Z2 charge of the fused index
  // (two halves: a quarter of the FP64 work); a connected matrix takes the plain tournament.
  for (int i = tid; i < n; i += nthr) comp[i] = i;
  __syncthreads();
  while (true) {
    int changed = 0;
    for (int e = tid; e < n * n; e += nthr) {
      const int i = e / n, j = e - i * n;
      if (i < j && nonzero(A[packed(i, j, n)])) {
        const int ci = comp[i], cj = comp[j];
        if (ci != cj) {
          atomicMin(&comp[ci < cj ? j : i], min(ci, cj));
          changed = 1;
        }
      }
    }
    if (!__syncthreads_or(changed)) break;
  }
  // components in the order of their smallest member; members in increasing index
  for (int i = tid; i < n; i += nthr) {
    int c = 0, pos = 0, size = 0;
    for (int j = 0; j < n; ++j) {
      c += comp[j] == j && j < comp[i];
      pos += comp[j] == comp[i] && j < i;
      size += comp[j] == comp[i];
    }
    cnum[i] = c;
    perm[i] = pos;                         // scratch: place inside the component
    if (comp[i] == i) sz[c] = size;
    if (i == n - 1) ncomp = 0;
  }
  __syncthreads();
  for (int i = tid; i < n; i += nthr)
    if (comp[i] == i) atomicAdd(&ncomp, 1);
  __syncthreads();
  const int nc = ncomp;
  for (int c = tid; c <= nc; c += nthr) {
    int b = 0, p = 0, t = 0, rm = 1, pm = 0;
    for (int k = 0; k < c; ++k) {
      const int np = (sz[k] + 1) / 2;
      b += sz[k];
      p += np;
      t += np * (np - 1) / 2;
      rm = max(rm, 2 * np - 1);
      pm = max(pm, np);
    }
    cbeg[c] = b;
    poff[c] = p;
    toff[c] = t;
    if (c == nc) {
      rmax = rm;
      npmax = pm;
    }
  }
  __syncthreads();
  for (int i = tid; i < n; i += nthr) mem[cbeg[cnum[i]] + perm[i]] = i;
  const int npairs = poff[nc], nblk = toff[nc], rounds = rmax;
  // 2x2 blocks off the diagonal (pair slots P < Q of one component), the same for every round
  for (int e = tid; e < nblk; e += nthr) {
    int c = 0;
    while (toff[c + 1] <= e) ++c;
    int P, Q;                              // the strict triangle of h slots is the triangle of h - 1
    tri_index(e - toff[c], poff[c + 1] - poff[c] - 1, P, Q);
    blk[e] = (uint32_t)(P + poff[c]) << 16 | (uint32_t)(Q + 1 + poff[c]);
  }
  // The last threads hold a pair slot each (warps of their own where there is room; npairs <= n <= threads): its
  // component, and its indices in the next round.
  const int slot = nthr - 1 - tid;
  int sc = 0;
  if (slot < npairs)
    while (poff[sc + 1] <= slot) ++sc;
  const int smc = cbeg[sc + 1] - cbeg[sc], smp = smc + (smc & 1), sb0 = cbeg[sc], sp0 = poff[sc];
  // indices (p < q) of slot sl of component c (m players, members from b) in round r; q = -1: none
  auto indices = [&](int r, int i, int mc, int mp, int b) {
    while (r >= mp - 1) r -= mp - 1;
    int lp, lq;
    rr_pair(r, i, mp, lp, lq);
    return make_short2((short)mem[b + lp], (short)(lq < mc ? mem[b + lq] : -1));
  };
  __syncthreads();
  short2 next = slot < npairs ? indices(0, slot - sp0, smc, smp, sb0) : make_short2(0, -1);
  // small matrices: a thread per entry of a 2x2 block (5 FP64 instructions instead of 13) where the CTA has them
  const int ws = nblk <= 40 && 4 * nblk + 32 <= nthr ? 2 : 0;

  // Applies the logged rotations in order to the rows of V (V <- V J), one row per warp.
  bool have_v = false;
  int nlog = 0;
  auto fold_log = [&]() {
    for (int row = tid >> 5; row < n; row += nthr >> 5) {
      double* v = V + (int64_t)row * n;
      if (!have_v)
        for (int j = lane; j < n; j += 32) v[j] = j == row ? 1.0 : 0.0;
      __syncwarp();
      for (int l = 0; l < nlog; ++l) {
        for (int sl = lane; sl < npairs; sl += 32) {
          const short2 i = logi[(int64_t)l * npairs + sl];
          if (i.y >= 0) {
            const double2 r = log[(int64_t)l * npairs + sl];
            const double vp = v[i.x], vq = v[i.y];
            v[i.x] = r.x * fma(-r.y, vq, vp);
            v[i.y] = r.x * fma(r.y, vp, vq);
          }
        }
        __syncwarp();
      }
    }
    have_v = true;
    nlog = 0;
    __syncthreads();
  };

  int sweep = 0;
  for (; sweep < max_sweeps && n > 1; ++sweep) {
    if (nlog + rounds > jobs.log_sweeps * n) fold_log();
    const int nlog0 = nlog;
    for (int r = 0; r < rounds; ++r) {
      int rot = 0;
      double cr = 1.0, tr = 0.0, app = 0, apq = 0, aqq = 0, d = 0;
      const short2 ij = next;
      if (slot < npairs) {
        const int p = ij.x, q = ij.y;
        if (q >= 0) {
          apq = A[packed(p, q, n)];
          app = A[packed(p, p, n)];
          aqq = A[packed(q, q, n)];
          if (rotates(apq, app, aqq)) {
            // tangent of the small rotation angle, t = 2 a_pq / (d + sign(d) sqrt(d^2 + 4 a_pq^2)), to FP32 accuracy
            // (any t gives an orthogonal rotation; the entry left over, 2^-22 of a_pq, goes with the next sweep), and
            // c = 1 / sqrt(1 + t^2) to FP64 accuracy from an FP32 start r by the binomial series of (1 - e)^(-1/2) =
            // 1 + e/2 + 3/8 e^2 + 5/16 e^3 + ..., 1 - e = (1 + t^2) r^2, |e| < 2^-20: two terms are enough
            d = aqq - app;
            const int ed = (__double2hiint(d) >> 20) & 0x7ff, eb = (__double2hiint(apq) >> 20) & 0x7ff;
            float tf;
            if (ed - eb > 60) {
              tr = apq / d;                   // below FP32's range
              tf = 0.0f;
            } else {
              const int em = max(ed, eb);     // largest magnitude to [1, 2)
              const float fd = scaled_float(d, em), fb = 2.0f * scaled_float(apq, em);
              tf = __fdividef(fb, fd + copysignf(__fsqrt_rn(fmaf(fd, fd, fb * fb)), fd));
              tr = widen(tf);
            }
            const double x = fma(tr, tr, 1.0);
            const double r0 = widen(rsqrtf(fmaf(tf, tf, 1.0f)));
            const double e = fma(-x, r0 * r0, 1.0);
            cr = fma(r0 * e, fma(e, 0.375, 0.5), r0);
            rot = 1;
          }
        }
        ct[slot] = make_double2(cr, tr);
        pq[slot] = ij;
        log[(int64_t)nlog * npairs + slot] = make_double2(cr, tr);
        logi[(int64_t)nlog * npairs + slot] = nonzero(tr) ? ij : make_short2(-1, -1);
      }
      const bool some = __syncthreads_or(rot);
      if (slot < npairs) next = indices(r + 1 < rounds ? r + 1 : 0, slot - sp0, smc, smp, sb0);
      if (!some) continue;   // nothing rotates in this round: its log entry is overwritten
      ++nlog;
      // A <- J^T A J: the rotated pairs' own blocks by the threads that hold the pairs, the blocks between two
      // pairs (P rows, Q columns) by the first threads
      if (nonzero(tr)) {
        // what is left of a_pq, r = (b (1 - t^2) - t (d - a)) c^2 (the difference keeps its error at 2^-52 of b), and
        // a' = a - t (b + r), d' = d + t (b + r)
        const double r = (cr * cr) * fma(-tr, tr * apq, fma(-tr, d, apq)), w = apq + r;
        A[packed(ij.x, ij.x, n)] = fma(-tr, w, app);
        A[packed(ij.y, ij.y, n)] = fma(tr, w, aqq);
        A[packed(ij.x, ij.y, n)] = r;
      }
      if (ws == 2) {
        if (tid - lane < 4 * nblk) {          // whole warps: the four threads of a block read before any writes
          const uint32_t PQ = blk[min(tid >> 2, nblk - 1)];
          const double2 r1 = ct[PQ >> 16], r2 = ct[PQ & 0xffffu];
          const short2 i1 = pq[PQ >> 16], i2 = pq[PQ & 0xffffu];
          const bool row = tid & 2, col = tid & 1;
          const bool hq1 = i1.y >= 0, hq2 = i2.y >= 0;
          const int p1 = i1.x, q1 = hq1 ? i1.y : p1, p2 = i2.x, q2 = hq2 ? i2.y : p2;
          // own row first: u, the other one: w
          const int ru = row ? q1 : p1, rw = row ? p1 : q1;
          const double up = A[packed(ru, p2, n)], uq = A[packed(ru, q2, n)];
          const double wp = hq1 ? A[packed(rw, p2, n)] : 0.0, wq = hq1 ? A[packed(rw, q2, n)] : 0.0;
          const double t1 = row ? r1.y : -r1.y, k = r1.x * r2.x;
          const double rp = fma(t1, wp, up), rq = hq2 ? fma(t1, wq, uq) : 0.0;
          const double v = k * (col ? fma(r2.y, rp, rq) : fma(-r2.y, rq, rp));
          __syncwarp();
          if (tid < 4 * nblk && (!row || hq1) && (!col || hq2)) A[packed(ru, col ? q2 : p2, n)] = v;
        }
        __syncthreads();
        continue;
      }
      for (int e = tid; e < nblk; e += nthr) {
        const uint32_t PQ = blk[e];
        const int P = (int)(PQ >> 16), Q = (int)(PQ & 0xffffu);
        const double2 r1 = ct[P], r2 = ct[Q];
        if (!nonzero(r1.y) && !nonzero(r2.y)) continue;
        const short2 i1 = pq[P], i2 = pq[Q];
        const int p1 = i1.x, q1 = i1.y, p2 = i2.x, q2 = i2.y;
        const bool hq1 = q1 >= 0, hq2 = q2 >= 0;
        const int ia = packed(p1, p2, n), ib = packed(p1, hq2 ? q2 : p2, n);
        const int ic = packed(hq1 ? q1 : p1, p2, n), id = packed(hq1 ? q1 : p1, hq2 ? q2 : p2, n);
        const double a = A[ia];
        const double b = hq2 ? A[ib] : 0.0;
        const double cc = hq1 ? A[ic] : 0.0;
        const double d = (hq1 && hq2) ? A[id] : 0.0;
        const double t1 = r1.y, t2 = r2.y, k = r1.x * r2.x;
        // rows, then columns, without the cosines
        const double ra = fma(-t1, cc, a), rb = fma(-t1, d, b);
        const double rc = fma(t1, a, cc), rd = fma(t1, b, d);
        const double na = k * fma(-t2, rb, ra), nd = k * fma(t2, rc, rd);
        const double nb = k * fma(t2, ra, rb), nc2 = k * fma(-t2, rd, rc);
        A[ia] = na;
        if (hq2) A[ib] = nb;
        if (hq1) A[ic] = nc2;
        if (hq1 && hq2) A[id] = nd;
      }
      __syncthreads();
    }
    if (nlog == nlog0) break;                 // nothing rotated
    // converged when no pair of a component would rotate
    int more = 0;
    for (int i = tid >> 5; i < n; i += nthr >> 5) {
      const int row = packed(i, i, n) - i;
      const double aii = A[row + i];
      for (int j = i + 1 + lane; j < n; j += 32)
        if (cnum[i] == cnum[j]) more |= rotates(A[row + j], aii, A[packed(j, j, n)]);
    }
    if (!__syncthreads_or(more)) {
      ++sweep;                                // a further sweep would find nothing to rotate
      break;
    }
  }
  if (tid == 0 && sweep >= max_sweeps && n > 1) atomicAdd(&status[kStNoConv], 1);

  // ---- sort descending (rank = number of larger eigenvalues, ties by index)
  // ranked by (value, index) as integers in the order of the values, a NaN as the lowest: a strict total order, so
  // perm is a permutation whatever the input (a non-finite tensor is reported by the normalisation)
  for (int i = tid; i < n; i += nthr) {
    const double v = A[packed(i, i, n)] * down;
    const long long b = __double_as_longlong(v);
    nrmv[i] = v;
    key[i] = (b & 0x7fffffffffffffffll) > 0x7ff0000000000000ll ? (long long)0x8000000000000000ull
                                                               : (b < 0 ? (long long)0x8000000000000000ull - b : b);
  }
  __syncthreads();
  for (int i = tid; i < n; i += nthr) {
    const long long ki = key[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += key[j] > ki || (key[j] == ki && j < i);
    perm[rank] = i;
    lam[rank] = nrmv[i];
  }
  __syncthreads();
  for (int i = tid; i < n; i += nthr) jb.lam[i] = lam[i];
  // clusters: start of the cluster each place belongs to (first thread of a place looks back)
  for (int j = tid; j < n; j += nthr) sz[j] = j == 0 || lam[j - 1] - lam[j] > cluster_tau * fabs(lam[0]);
  __syncthreads();
  for (int j = tid; j <= n; j += nthr) {
    int k = 0;
    for (int i = 0; i < j; ++i) k += sz[i];
    if (j == n) {
      cstart[k] = n;
      ncl = k;
    } else if (sz[j]) {
      cstart[k] = j;
    }
  }
  // the discarded sum: each lane of the first warp its share, then pairwise
  if (tid < 32) {
    double e = 0;
    for (int j = chi + lane; j < n; j += 32) e += lam[j];
    for (int off = 16; off > 0; off >>= 1) e += __shfl_xor_sync(0xffffffffu, e, off);
    if (tid == 0) *jb.eps = e;
  }
  __syncthreads();
  // columns needed: every member of a cluster that starts below chi
  int nw = chi;
  while (nw < n && !sz[nw]) ++nw;
  if (tid == 0) *jb.degenerate = nw > chi;     // the cut falls inside a cluster

  // ---- eigenvectors: columns perm[0 .. nw) of V = J_1 J_2 ... J_m, from the unit vectors with the last rotation
  // first. A column lives in the indices of its component; gsz lanes hold its pairs.
  {
    int gsz = 1;
    while (gsz < npmax && gsz < 32) gsz *= 2;
    const int par = min(nthr / gsz, region / n);       // columns at a time
    const int gid = tid / gsz, lg = tid - gid * gsz;
    const bool one = npmax <= gsz;                     // a lane holds at most one pair
    for (int k0 = 0; k0 < nw; k0 += par) {
      const int k = k0 + gid;
      const bool live = gid < par && k < nw;
      double* w = dyn + (int64_t)(live ? gid : 0) * n;
      const int col = live ? perm[k] : 0, c = cnum[col];
      const int np = (cbeg[c + 1] - cbeg[c] + 1) / 2, p0 = poff[c];
      if (live)
        for (int j = lg; j < n; j += gsz) w[j] = j == col ? 1.0 : 0.0;
      __syncwarp();
      auto apply = [&](short2 i, double2 r) {
        if (i.y >= 0) {
          const double wp = w[i.x], wq = w[i.y];
          w[i.x] = r.x * fma(r.y, wq, wp);
          w[i.y] = r.x * fma(-r.y, wp, wq);
        }
      };
      if (one) {
        // four entries ahead: their rotations and indices are read before the column's own chain needs them
        const bool act = live && lg < np;
        const double2* lr = log + p0 + lg;
        const short2* li = logi + p0 + lg;
        double2 nr[4];
        short2 ni[4];
        auto fetch = [&](int l, int u) {
          const bool in = act && l >= 0;
          ni[u] = in ? li[(int64_t)l * npairs] : make_short2(-1, -1);
          nr[u] = in ? lr[(int64_t)l * npairs] : make_double2(1.0, 0.0);
        };
#pragma unroll
        for (int u = 0; u < 4; ++u) fetch(nlog - 1 - u, u);
        for (int l = nlog - 1; l >= 0; l -= 4) {
          double2 r[4];
          short2 ij[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            r[u] = nr[u];
            ij[u] = ni[u];
            fetch(l - 4 - u, u);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            apply(ij[u], r[u]);
            __syncwarp();
          }
        }
      } else {
        for (int l = nlog - 1; l >= 0; --l) {
          if (live)
            for (int sl = lg; sl < np; sl += gsz)
              apply(logi[(int64_t)l * npairs + p0 + sl], log[(int64_t)l * npairs + p0 + sl]);
          __syncwarp();
        }
      }
      if (live)
        for (int j = lg; j < n; j += gsz) {
          double v = w[j];
          if (have_v) {                                // V J_log e = V w
            v = 0;
            for (int i = 0; i < n; ++i) v = fma(V[(int64_t)j * n + i], w[i], v);
          }
          W[(int64_t)k * n + j] = v;
        }
      __syncwarp();
    }
  }
  __threadfence_block();
  __syncthreads();

  // ---- canonical gauge for the first chi columns, written to U (n x chi): one warp per cluster
  for (int c = tid >> 5; c < ncl; c += nthr >> 5) {
    const int s0 = cstart[c], e0 = cstart[c + 1];
    if (s0 >= chi) break;
    if (e0 == s0 + 1) {
      // a simple eigenvalue: the sign that makes its pivot component positive
      const double* w = W + (int64_t)s0 * n;
      double mx = 0;
      for (int i = lane; i < n; i += 32) mx = fmax(mx, w[i] * w[i]);
      for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      int ip = n;
      for (int i = lane; i < n && ip == n; i += 32)
        if (w[i] * w[i] >= (1.0 - tie_rel) * mx) ip = i;
      for (int off = 16; off > 0; off >>= 1) ip = min(ip, __shfl_xor_sync(0xffffffffu, ip, off));
      const double sg = ip < n && w[ip] < 0 ? -1.0 : 1.0;
      for (int i = lane; i < n; i += 32) jb.U[i * chi + s0] = sg * w[i];
      continue;
    }
    // nrm = |P_cluster e_i|^2 minus what the columns so far cover; each lane keeps its own indices
    double nr[kMaxGramN / 32];
#pragma unroll
    for (int t = 0; t < kMaxGramN / 32; ++t) {
      const int i = lane + 32 * t;
      double b = 0;
      if (i < n)
        for (int j = s0; j < e0; ++j) {
          const double v = W[(int64_t)j * n + i];
          b = fma(v, v, b);
        }
      nr[t] = b;
    }
    const int tend = min(e0, chi);
    for (int t = s0; t < tend; ++t) {
      double mx = 0;
#pragma unroll
      for (int u = 0; u < kMaxGramN / 32; ++u)
        if (lane + 32 * u < n) mx = fmax(mx, nr[u]);
      for (int off = 16; off > 0; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      int ip = n;
      double pv = 0;
#pragma unroll
      for (int u = kMaxGramN / 32 - 1; u >= 0; --u)
        if (lane + 32 * u < n && nr[u] >= (1.0 - tie_rel) * mx) {
          ip = lane + 32 * u;
          pv = nr[u];
        }
      int best = ip;
      for (int off = 16; off > 0; off >>= 1) best = min(best, __shfl_xor_sync(0xffffffffu, best, off));
      if (best >= n) best = 0;                 // NaN: any index in range (the norm reports the tensor)
      pv = __shfl_sync(0xffffffffu, pv, best & 31);
      const double inv = 1.0 / sqrt(pv);
#pragma unroll
      for (int u = 0; u < kMaxGramN / 32; ++u) {
        const int i = lane + 32 * u;
        if (i < n) {
          double g = 0;
          for (int j = s0; j < e0; ++j) g = fma(W[(int64_t)j * n + i], W[(int64_t)j * n + best], g);
          for (int v = s0; v < t; ++v) g -= jb.U[i * chi + v] * jb.U[best * chi + v];
          g *= inv;
          nr[u] -= g * g;
          jb.U[i * chi + t] = g;
        }
      }
      __threadfence_block();
      __syncwarp();
    }
  }
}

// The shared-memory attribute is set once per device: by jacobi_prepare (called when a
// workspace is attached, ahead of any stream capture) or at the first launch on a device.
constexpr int kJacobiMaxDevices = 64;
bool g_jacobi_attr[kJacobiMaxDevices] = {};

// Dynamic shared memory: region doubles for A (or the columns in progress), and the block list.
struct JacobiSmem {
  int region;
  size_t bytes;
};
JacobiSmem jacobi_smem(int nmax) {
  const int np = (nmax + 1) / 2;
  const int cols = (kJT / 32) * nmax;          // 17 columns in progress
  JacobiSmem s;
  s.region = nmax <= kJacobiSmemN ? (int)packed_doubles(nmax) : cols;
  const int blocks = np * (np - 1) / 2 + 1;    // of a connected matrix: components have fewer in all
  s.bytes = (size_t)s.region * sizeof(double) + (size_t)blocks * sizeof(uint32_t);
  return s;
}

cudaError_t jacobi_attr_for_current_device() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kJacobiMaxDevices) return cudaErrorInvalidDevice;
  if (g_jacobi_attr[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(jacobi_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)jacobi_smem(kJacobiSmemN).bytes);
  if (e == cudaSuccess) g_jacobi_attr[dev] = true;
  return e;
}

void jacobi_prepare() { jacobi_attr_for_current_device(); }

cudaError_t launch_jacobi(const EigPack& jobs, int njobs, int nmax, double cluster_tau, int* status,
                          cudaStream_t st, int max_sweeps, double tie_rel) {
  if (nmax < 1 || nmax > kMaxGramN) return cudaErrorInvalidValue;
  const JacobiSmem sm = jacobi_smem(nmax);
  const cudaError_t e = jacobi_attr_for_current_device();
  if (e != cudaSuccess) return e;
  // a thread per 2x2 block of a connected matrix, up to kJT: whole warps of blocks between pairs and of pairs
  const int np = (nmax + 1) / 2, want = (np * (np - 1) / 2 + 31) / 32 * 32 + (np + 31) / 32 * 32;
  const int threads = want < 192 ? 192 : (want > kJT ? kJT : want);   // at least nmax: np^2 / 2 + 32 > 2 np from 192 on
  jacobi_kernel<<<njobs * jobs.batch, threads, sm.bytes, st>>>(jobs, njobs, nmax <= kJacobiSmemN ? 1 : 0, sm.region,
                                                              cluster_tau, tie_rel, max_sweeps, status);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------- side choice
template <typename R>
__global__ void __launch_bounds__(256) select_kernel(const __grid_constant__ SelectPack jobs, int njobs,
                                                     double side_rel) {
  // job blockIdx.x % njobs of batch element blockIdx.x / njobs
  const int64_t bidx = blockIdx.x / njobs;
  SelectJob jb = jobs.j[blockIdx.x - bidx * njobs];
  jb.U[0] += bidx * jobs.sU;
  jb.U[1] += bidx * jobs.sU;
  jb.lam0 += bidx * jobs.sLam;
  jb.eps[0] += bidx * jobs.sEps;
  jb.eps[1] += bidx * jobs.sEps;
  jb.degen[0] += bidx * jobs.sDeg;
  jb.degen[1] += bidx * jobs.sDeg;
  jb.U64 += bidx * jobs.sU64;
  jb.Ur = (R*)jb.Ur + bidx * jobs.sUr;
  if (jb.rec_b) jb.rec_b += bidx * jobs.sRec;
  if (jb.sectors) jb.sectors += bidx;
  __shared__ int seen[kMaxLeg];      // charges met in each kept column (bit 0: even, bit 1: odd)
  __shared__ double Q[4096];         // columns of n: n chi <= 256 x 16, 64 x 64
  __shared__ int side;
  const int n = jb.n, chi = jb.chi, tid = threadIdx.x;
  if (tid == 0) {
    const double e0 = *jb.eps[0], e1 = *jb.eps[1];
    side = (e0 - e1 > side_rel * (fabs(e0) + fabs(e1)) + 1e-13 * fabs(jb.lam0[0])) ? 1 : 0;
    double* re = jb.rec_eps;
    int* rp = jb.rec_primed;
    int* rd = jb.rec_degen;
    if (jb.rec_b != nullptr) {           // record slot of the current step, read on the device
      const int k = *jb.step < kMaxSteps ? *jb.step : kMaxSteps - 1;
      re = jb.rec_b[k].eps[jb.nu];
      rp = &jb.rec_b[k].primed[jb.nu];
      rd = &jb.rec_b[k].degen[jb.nu];
    }
    re[0] = e0;
    re[1] = e1;
    *rp = side;
    *rd = *jb.degen[side];
  }
  __syncthreads();
  // modified Gram-Schmidt in FP64, in shared memory: column j normalised by one warp, then taken out of
  // every later column, one warp per column (for each column the same steps in the same order)
  const double* src = jb.U[side];
  const int lane = tid & 31, wid = tid >> 5;
  for (int e = tid; e < n * chi; e += blockDim.x) Q[e % chi * n + e / chi] = src[e];
  __syncthreads();
  for (int j = 0; j < chi; ++j) {
    double* uj = Q + j * n;
    if (wid == 0) {
      double q = 0;
      for (int r = lane; r < n; r += 32) q = fma(uj[r], uj[r], q);
      for (int off = 16; off > 0; off >>= 1) q += __shfl_xor_sync(0xffffffffu, q, off);
      const double inv = rsqrt(q);
      for (int r = lane; r < n; r += 32) uj[r] *= inv;
    }
    __syncthreads();
    for (int k = j + 1 + wid; k < chi; k += blockDim.x >> 5) {
      double* uk = Q + k * n;
      double d = 0;
      for (int r = lane; r < n; r += 32) d = fma(uj[r], uk[r], d);
      for (int off = 16; off > 0; off >>= 1) d += __shfl_xor_sync(0xffffffffu, d, off);
      for (int r = lane; r < n; r += 32) uk[r] -= d * uj[r];
    }
    __syncthreads();
  }
  for (int e = tid; e < n * chi; e += blockDim.x) jb.U64[e] = Q[e % chi * n + e / chi];
  R* ur = (R*)jb.Ur;
  for (int e = tid; e < n * chi; e += blockDim.x) ur[e] = (R)Q[e % chi * n + e / chi];
  if (jb.sectors == nullptr) return;
  // charge of a kept column = charge of the fused indices it is made of; a column that mixes both
  // drops the element's sectors
  for (int i = tid; i < chi; i += blockDim.x) seen[i] = 0;
  __syncthreads();
  const uint32_t m = jb.sectors->charge[jb.cur][jb.nu];
  for (int e = tid; e < n * chi; e += blockDim.x)
    if (Q[e % chi * n + e / chi] != 0.0) {
      const int r = e / chi;
      atomicOr(&seen[e % chi], 1 << (((m >> (r / jb.Dn)) ^ (m >> (r % jb.Dn))) & 1));
    }
  __syncthreads();
  if (tid == 0) {
    uint32_t q = 0;
    for (int i = 0; i < chi; ++i) {
      if (seen[i] == 3) jb.sectors->dropped = 1;
      if (seen[i] == 2) q |= 1u << i;
    }
    jb.sectors->charge[1 - jb.cur][jb.nu] = q;
    if (blockIdx.x - bidx * njobs == 0) jb.sectors->charge[1 - jb.cur][jb.mu] = jb.sectors->charge[jb.cur][jb.mu];
  }
}

template <typename R>
cudaError_t launch_select(const SelectPack& jobs, int njobs, double side_rel, cudaStream_t st) {
  select_kernel<R><<<njobs * jobs.batch, 256, 0, st>>>(jobs, njobs, side_rel);
  return cudaGetLastError();
}
template cudaError_t launch_select<double>(const SelectPack&, int, double, cudaStream_t);
template cudaError_t launch_select<float>(const SelectPack&, int, double, cudaStream_t);

}  // namespace hotrg
