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
// The FP64 pipe (a warp instruction every 16 cycles per SM) and the latency of a round bound it.
// So A is kept as its upper triangle (16 FP64 instructions per 2x2 block on or above the
// diagonal, nothing mirrored), the rotation costs two reciprocal square roots, a round in which
// nothing rotates is skipped, and the eigenvector matrix is not accumulated: the rotations are
// logged, and the columns that are needed (the clusters that reach into the first chi; 8 of 64 at
// D = 8) are formed at the end by applying the log backwards to unit vectors, one column per
// group of lanes without block barriers.
//
// select_kernel: per transverse direction, the side (nu or nu') with the smaller
// discarded sum (a difference within side_rel (eps + eps') + 1e-13 lambda_0 is a tie and
// goes to nu; side_rel = 1e-9 for FP64 tensors, 1e-6 for FP32 ones), then modified Gram-Schmidt in FP64 on the kept vectors, and copies of U in
// FP64 and in the storage precision.
#include <math.h>

#include "common.cuh"

namespace hotrg {

constexpr int kJT = 544;            // most threads of a Jacobi CTA: the 528 blocks of n = 64 in one pass

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

__device__ double block_sum(double v, double* red) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
  __syncthreads();
  return s;
}


// Place of entry (i, j) in the packed upper triangle of an n x n matrix.
__device__ __forceinline__ int packed(int i, int j, int n) {
  const int lo = min(i, j), hi = max(i, j);
  return lo * (2 * n - 1 - lo) / 2 + hi;
}

__global__ void __launch_bounds__(kJT) jacobi_kernel(const __grid_constant__ EigPack jobs, int njobs, int use_smem,
                                                     int region, double cluster_tau, double tie_rel, int max_sweeps,
                                                     int* status) {
  extern __shared__ double dyn[];          // region doubles (A, later the columns in progress), then the block list
  // one slot per rotation pair of a round: at most n (ceil(m_c / 2) <= m_c per component)
  __shared__ double cs[kMaxGramN], sn[kMaxGramN];
  __shared__ short pp[kMaxGramN], qq[kMaxGramN];
  __shared__ double lam[kMaxGramN], nrm[kMaxGramN];
  __shared__ int perm[kMaxGramN], cstart[kMaxGramN + 1];
  __shared__ double red[kJT / 32];
  __shared__ int comp[kMaxGramN];          // component label: its smallest index
  __shared__ int cnum[kMaxGramN];          // component number of an index
  __shared__ int mem[kMaxGramN];           // indices grouped by component
  __shared__ int cbeg[kMaxGramN + 1];      // component c: mem[cbeg[c] .. cbeg[c + 1])
  __shared__ int poff[kMaxGramN + 1];      // first pair slot of component c
  __shared__ int toff[kMaxGramN + 1];      // first 2x2 block of component c
  __shared__ int sz[kMaxGramN];
  __shared__ unsigned char lround[kJacobiLogSweeps * kMaxGramN];   // round of each log entry
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
  double* A = use_smem ? dyn : Aw;         // use_smem: every job of the launch has n <= kJacobiSmemN
  uint32_t* blk = (uint32_t*)(dyn + region);

  // the upper triangle of G (the merged Gram is symmetric up to summation order), scaled by a power
  // of two to a largest magnitude in [1, 2), so that squares neither overflow nor vanish
  double big = 0;
  for (int e = tid; e < n * n; e += nthr) {
    const int i = e / n, j = e - i * n;
    if (i <= j) big = fmax(big, fabs(jb.G[e]));
  }
  for (int off = 16; off > 0; off >>= 1) big = fmax(big, __shfl_down_sync(0xffffffffu, big, off));
  if (lane == 0) red[tid >> 5] = big;
  __syncthreads();
  big = 0;
  for (int w = 0; w < nthr >> 5; ++w) big = fmax(big, red[w]);
  __syncthreads();
  const int sh = big > 0 && big < INFINITY ? ilogb(big) : 0;
  const double up = ldexp(1.0, sh < -1000 ? 1000 : (sh > 1000 ? -1000 : -sh)), down = 1.0 / up;   // exact
  double fro = 0;
  for (int e = tid; e < n * n; e += nthr) {
    const int i = e / n, j = e - i * n;
    if (i > j) continue;
    const double g = jb.G[e] * up;
    A[packed(i, j, n)] = g;
    fro = fma(i == j ? g : 2 * g, g, fro);
  }
  fro = sqrt(block_sum(fro, red));
  const double tol_abs = 1e-18 * fro;
  const double tol2 = 2.220446049250313e-16 * 2.220446049250313e-16;
  auto rotates = [&](double apq, double app, double aqq) {
    return fabs(apq) > tol_abs && apq * apq > tol2 * fabs(app * aqq);
  };

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
      if (i < j && A[packed(i, j, n)] != 0.0) {
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
      t += np * (np + 1) / 2;
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
  // 2x2 blocks (pair slots P <= Q of one component), the same for every round
  for (int e = tid; e < nblk; e += nthr) {
    int c = 0;
    while (toff[c + 1] <= e) ++c;
    int P, Q;
    tri_index(e - toff[c], poff[c + 1] - poff[c], P, Q);
    blk[e] = (uint32_t)(P + poff[c]) << 16 | (uint32_t)(Q + poff[c]);
  }
  // this thread's first pair slot
  int sc = 0;
  if (tid < npairs)
    while (poff[sc + 1] <= tid) ++sc;
  __syncthreads();

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
          int c = 0;
          while (poff[c + 1] <= sl) ++c;
          const int mc = cbeg[c + 1] - cbeg[c], mp = mc + (mc & 1);
          int lp, lq;
          rr_pair(lround[l] % (mp - 1), sl - poff[c], mp, lp, lq);
          if (lq < mc) {
            const double2 r = log[(int64_t)l * npairs + sl];
            const int p = mem[cbeg[c] + lp], q = mem[cbeg[c] + lq];
            const double vp = v[p], vq = v[q];
            v[p] = r.x * vp - r.y * vq;
            v[q] = r.y * vp + r.x * vq;
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
    if (nlog + rounds > kJacobiLogSweeps * n) fold_log();
    const int nlog0 = nlog;
    for (int r = 0; r < rounds; ++r) {
      int rot = 0;
      for (int sl = tid; sl < npairs; sl += nthr) {
        int c = sc;
        if (sl != tid) {
          c = 0;
          while (poff[c + 1] <= sl) ++c;
        }
        const int mc = cbeg[c + 1] - cbeg[c], mp = mc + (mc & 1);
        int rr = r;
        while (rr >= mp - 1) rr -= mp - 1;
        int lp, lq;
        rr_pair(rr, sl - poff[c], mp, lp, lq);
        const int p = mem[cbeg[c] + lp], q = lq < mc ? mem[cbeg[c] + lq] : -1;
        double cr = 1.0, sr = 0.0;
        if (q >= 0) {
          const double apq = A[packed(p, q, n)], app = A[packed(p, p, n)], aqq = A[packed(q, q, n)];
          if (rotates(apq, app, aqq)) {
            // the small rotation angle theta, tan 2 theta = 2 a_pq / (a_qq - a_pp): cos 2 theta = |d| / h >= 0,
            // c = sqrt((1 + cos 2 theta) / 2), s = sin 2 theta / (2 c); two reciprocal square roots on the
            // round's critical path
            const double d = aqq - app, t = 2.0 * apq;
            const double ih = rsqrt(fma(d, d, t * t));
            const double u = fma(0.5 * fabs(d), ih, 0.5);
            const double ic = rsqrt(u);
            cr = u * ic;
            sr = (d >= 0 ? apq : -apq) * ih * ic;
            rot = 1;
          }
        }
        cs[sl] = cr;
        sn[sl] = sr;
        pp[sl] = (short)p;
        qq[sl] = (short)q;
        log[(int64_t)nlog * npairs + sl] = make_double2(cr, sr);
      }
      if (tid == 0) lround[nlog] = (unsigned char)r;
      if (!__syncthreads_or(rot)) continue;   // nothing rotates in this round: its log entry is overwritten
      ++nlog;
      // A <- J^T A J, one 2x2 block (pair P rows, pair Q columns) per thread iteration
      for (int e = tid; e < nblk; e += nthr) {
        const uint32_t PQ = blk[e];
        const int P = (int)(PQ >> 16), Q = (int)(PQ & 0xffffu);
        const double c1 = cs[P], s1 = sn[P], c2 = cs[Q], s2 = sn[Q];
        if (s1 == 0.0 && s2 == 0.0) continue;
        const int p1 = pp[P], q1 = qq[P], p2 = pp[Q], q2 = qq[Q];
        const bool hq1 = q1 >= 0, hq2 = q2 >= 0;
        const int ia = packed(p1, p2, n), ib = packed(p1, hq2 ? q2 : p2, n);
        const int ic = packed(hq1 ? q1 : p1, p2, n), id = packed(hq1 ? q1 : p1, hq2 ? q2 : p2, n);
        const double a = A[ia];
        const double b = hq2 ? A[ib] : 0.0;
        const double cc = hq1 ? A[ic] : 0.0;
        const double d = (hq1 && hq2) ? A[id] : 0.0;
        // rows
        const double ra = c1 * a - s1 * cc, rb = c1 * b - s1 * d;
        const double rc = s1 * a + c1 * cc, rd = s1 * b + c1 * d;
        // columns
        const double na = c2 * ra - s2 * rb, nd = s2 * rc + c2 * rd;
        double nb = s2 * ra + c2 * rb, nc2 = c2 * rc - s2 * rd;
        if (P == Q) nb = nc2 = 0.0;           // the rotated pair (s1 != 0 here)
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
    for (int e = tid; e < n * n; e += nthr) {
      const int i = e / n, j = e - i * n;
      if (i < j && cnum[i] == cnum[j]) more |= rotates(A[packed(i, j, n)], A[packed(i, i, n)], A[packed(j, j, n)]);
    }
    if (!__syncthreads_or(more)) {
      ++sweep;                                // a further sweep would find nothing to rotate
      break;
    }
  }
  if (tid == 0 && sweep >= max_sweeps && n > 1) atomicAdd(&status[kStNoConv], 1);

  // ---- sort descending (rank = number of larger eigenvalues, ties by index)
  for (int i = tid; i < n; i += nthr) nrm[i] = A[packed(i, i, n)] * down;
  __syncthreads();
  for (int i = tid; i < n; i += nthr) {
    // ranked by (value, index) with a NaN taken as -inf: a strict total order, so perm is a
    // permutation whatever the input (a non-finite tensor is reported by the normalisation)
    const double li = nrm[i], ki = li == li ? li : -INFINITY;
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double lj = nrm[j], kj = lj == lj ? lj : -INFINITY;
      rank += (kj > ki) || (kj == ki && j < i);
    }
    perm[rank] = i;
    lam[rank] = li;
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
  // the discarded sum, in decreasing order
  if (tid == 0) {
    double e = 0;
    for (int j = chi; j < n; ++j) e += lam[j];
    *jb.eps = e;
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
      const int mc = cbeg[c + 1] - cbeg[c], mp = mc + (mc & 1), np = mp / 2, p0 = poff[c], b0 = cbeg[c];
      if (live)
        for (int j = lg; j < n; j += gsz) w[j] = j == col ? 1.0 : 0.0;
      __syncwarp();
      auto apply = [&](int l, int sl, double2 r) {
        int rr = lround[l];
        while (rr >= mp - 1) rr -= mp - 1;
        int lp, lq;
        rr_pair(rr, sl, mp, lp, lq);
        if (lq < mc && r.y != 0.0) {
          const int p = mem[b0 + lp], q = mem[b0 + lq];
          const double wp = w[p], wq = w[q];
          w[p] = r.x * wp + r.y * wq;
          w[q] = r.x * wq - r.y * wp;
        }
      };
      if (one) {
        const bool act = live && lg < np;
        const double2* lp0 = log + p0 + lg;
        double2 nx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          nx[u] = act && nlog - 1 - u >= 0 ? lp0[(int64_t)(nlog - 1 - u) * npairs] : make_double2(1.0, 0.0);
        for (int l = nlog - 1; l >= 0; l -= 4) {
          double2 cur[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            cur[u] = nx[u];
            nx[u] = act && l - 4 - u >= 0 ? lp0[(int64_t)(l - 4 - u) * npairs] : make_double2(1.0, 0.0);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (act && l - u >= 0) apply(l - u, lg, cur[u]);
            __syncwarp();
          }
        }
      } else {
        for (int l = nlog - 1; l >= 0; --l) {
          if (live)
            for (int sl = lg; sl < np; sl += gsz) apply(l, sl, log[(int64_t)l * npairs + p0 + sl]);
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
  // blocks: at most one more than a connected matrix has (components of n - 1 and 1), or one per index
  const int blocks = np * (np + 1) / 2 + 1 > nmax ? np * (np + 1) / 2 + 1 : nmax;
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
  // a thread per 2x2 block of a connected matrix, up to kJT
  const int np = (nmax + 1) / 2, want = (np * (np + 1) / 2 + 31) / 32 * 32;
  const int threads = want < 64 ? 64 : (want > kJT ? kJT : want);
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
      const double inv = 1.0 / sqrt(q);
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
