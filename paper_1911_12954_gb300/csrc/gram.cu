// gram.cu - Gram (environment) matrices of the HOSVD of two adjacent tensors (Fig. 1B).
//
// For a step along mu and a transverse leg l (nu or nu'), the Gram matrix of the pair
// tensor M = T1 -mu- T2 on its fused (T1.l, T2.l) leg factorises into two half-Grams of
// the single tensor, each a symmetric rank-K update with rows (l, mu-leg):
//   A1[(a,k),(b,k')] = sum_rest T[a@l, k@mu', rest] T[b@l, k'@mu', rest]
//   A2[(a,k),(b,k')] = sum_rest T[a@l, k@mu , rest] T[b@l, k'@mu , rest]
//   G[(a1 a2),(b1 b2)] = sum_{k,k'} A1[(a1,k),(b1,k')] A2[(a2,k),(b2,k')].
// gram_kernel computes upper-triangle tiles (64 x 64 at most) of one half-Gram over one chunk of
// the summed index (split-K: K = D^6 is long, R = D_l D_mu is short), products in the storage
// precision summed with FMA over slices of a few terms, then the slice sums accumulated: in
// FP64 for FP64 tensors, for FP32 ones as an unevaluated pair of floats (hi + lo, Knuth's TwoSum)
// that adds them without a further rounding and without the FP64 pipe (a few FP64 operations
// per clock per SM on this chip, against 128 FP32 FMAs). For FP32 tensors a slice is 8 terms: its
// rounding errors are a few 2^-24 of the slice's magnitude, whatever K is, where one FP32 running
// sum over K = D^6 terms would add an error that grows with K (the error of sums of one sign
// is proportional to the slice's length; the pair sums cost 7 instructions per 8 FMAs).
// gram_reduce adds the chunks of every job in a fixed order (deterministic, one launch);
// gram_merge forms G in FP64.
//
// The FMAs bound it (FP64: the FP64 pipe, 16 cycles per warp instruction). So only blocks on or
// above the diagonal are computed, R is not padded to the tile (R = 16 at D = 4), and where the
// tensor conserves the Z2 charge (SectorState) rows meet only the summed indices of their own
// charge: two problems of half the rows over half the indices, a quarter of the FMAs. A thread owns
// a 4 x 4 block; blocks that do not fill the CTA are taken by several thread groups, each
// summing every G-th index of a slab. FP64: 288 threads, one CTA per SM (2 x 136 triangle blocks
// at R = 64 fill the FP64 pipe: 91 % busy on 64 x 64 rows); FP32: 256 threads, two CTAs per SM to cover the loads.
#include <type_traits>

#include "common.cuh"

namespace hotrg {

constexpr int kGT = 64;          // rows of a tile
template <typename R>
constexpr int kGramThreads = sizeof(R) == 8 ? 288 : 256;
constexpr int kGList = 2048;     // summed indices decoded at once
constexpr int kGBuf = 4608;      // elements of the operand slab (two slabs of 32 x 68 off the diagonal)
constexpr int kGLoad = 8;        // slab elements per thread: at most 2048 per slab

// hi + lo += x exactly up to the rounding of lo (TwoSum of hi and x).
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x) {
  const float t = hi + x;
  const float bp = t - hi;
  const float err = (hi - (t - bp)) + (x - bp);
  hi = t;
  lo += err;
}

// Masks (charges) of the row legs and of one summed leg; 0 where the tensor keeps none.
__device__ __forceinline__ uint32_t gram_mask(const GramPack& p, int bidx, int dir) {
  if (!p.sectors) return 0u;
  const SectorState& s = p.sectors[bidx];
  return s.dropped ? 0u : s.charge[p.cur][dir];
}
__device__ __forceinline__ int odd_count(uint32_t m, int n) { return __popc(m & ((1u << n) - 1u)); }

template <typename R>
__global__ void __launch_bounds__(kGramThreads<R>, sizeof(R) == 8 ? 1 : 2)
    gram_kernel(const __grid_constant__ GramPack jobs, int njobs, int nchunks) {
  constexpr int kGThreads = kGramThreads<R>;
  const int bidx = blockIdx.z / njobs;        // batch element
  const GramJob& jb = jobs.j[blockIdx.z - bidx * njobs];
  const int Rn = jb.D1 * jb.D2;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint32_t m1 = gram_mask(jobs, bidx, jb.dir1), m2 = gram_mask(jobs, bidx, jb.dir2);
  // rows of charge 0 and 1; tile pairs (ti <= tj) of charge 0, then of charge 1
  const int o1 = odd_count(m1, jb.D1), o2 = odd_count(m2, jb.D2);
  const int R1 = o1 * (jb.D2 - o2) + (jb.D1 - o1) * o2, R0 = Rn - R1;
  const int nt0 = (R0 + kGT - 1) / kGT, nt1 = (R1 + kGT - 1) / kGT;
  int pr = blockIdx.y, q = 0;
  if (pr >= nt0 * (nt0 + 1) / 2) {
    pr -= nt0 * (nt0 + 1) / 2;
    q = 1;
  }
  const int nt = q ? nt1 : nt0, Rq = q ? R1 : R0;
  if (pr >= nt * (nt + 1) / 2) return;
  int ti = 0;
  while (pr >= nt - ti) pr -= nt - ti++;
  const int tj = ti + pr;
  const bool diag = ti == tj;                 // both operand tiles are the same rows
  const int ni = min(kGT, Rq - ti * kGT), nj = min(kGT, Rq - tj * kGT);
  const R* T = (const R*)jb.T + bidx * jobs.sT;
  const int64_t kchunk = (jb.K + nchunks - 1) / nchunks;
  const int64_t k0 = blockIdx.x * kchunk;
  const int64_t k1 = min(jb.K, k0 + kchunk);

  __shared__ __align__(16) R X[kGBuf];
  __shared__ uint32_t list[kGList];           // offsets of the summed indices of charge q
  __shared__ uint32_t roff[2][kGT];           // offsets of the tile's rows, and their places in the output
  __shared__ uint16_t rout[2][kGT];
  __shared__ int wcnt[8 * (kGThreads / 32) + 1];

  // rows in the order (slower leg, faster leg): neighbours in memory are neighbours in the tile
  {
    const bool swap = jb.s1 < jb.s2;          // leg 1 is the faster one
    const int Ds = swap ? jb.D2 : jb.D1, Df = swap ? jb.D1 : jb.D2;
    const uint32_t ms = swap ? m2 : m1, mf = swap ? m1 : m2;
    const int of = odd_count(mf, Df);
    for (int r = tid; r < Rn; r += kGThreads) {
      const int is = r / Df, f = r - is * Df;
      const int qs = (ms >> is) & 1;
      if ((qs ^ ((mf >> f) & 1)) != q) continue;
      const int so = odd_count(ms, is), se = is - so;      // slower indices before, by charge
      const int fo = odd_count(mf, f);
      const int rank = (q ? se * of + so * (Df - of) : se * (Df - of) + so * of) + ((q ^ qs) ? fo : f - fo);
      const int i1 = swap ? f : is, i2 = swap ? is : f;
      const uint32_t off = (uint32_t)(i1 * jb.s1 + i2 * jb.s2);
      const uint16_t out = (uint16_t)(i1 * jb.D2 + i2);
      if (rank / kGT == ti) {
        roff[0][rank - ti * kGT] = off;
        rout[0][rank - ti * kGT] = out;
      }
      if (rank / kGT == tj) {
        roff[1][rank - tj * kGT] = off;
        rout[1][rank - tj * kGT] = out;
      }
    }
    (void)Ds;
  }
  // 4 x 4 blocks of the tile (the triangle on the diagonal), G thread groups over the slab's indices
  const int bi_n = (ni + 3) / 4, bj_n = (nj + 3) / 4;
  const int nblk = diag ? bi_n * (bi_n + 1) / 2 : bi_n * bj_n;
  const int G = kGThreads / nblk;
  const int g = tid / nblk;
  int bi, bj;
  if (diag) {
    int e = tid - g * nblk;
    bi = 0;
    while (e >= bi_n - bi) e -= bi_n - bi++;
    bj = bi + e;
  } else {
    const int e = tid - g * nblk;
    bi = e / bj_n;
    bj = e - bi * bj_n;
  }
  const bool works = g < G;
  // slab: KS indices x the tile's rows, pitch = 4 (mod 32) words: the loads below take 8 indices x 4 rows per
  // warp (whole 32-byte sectors) and store them without bank conflicts
  const int ri = 4 * bi_n, rj = 4 * bj_n, rm = diag ? ri : max(ri, rj);
  const int pitch = (rm + 31) / 32 * 32 + 4;
  int KS = 2048 / (diag ? ri : ri + rj) / 8 * 8;
  KS = min(KS, kGBuf / (diag ? pitch : 2 * pitch) / 8 * 8);
  KS = min(KS, 128);
  // whole slices of 8 terms per group where the slab has room for them
  const bool whole = 8 * G <= KS;
  if (whole) KS = KS / (8 * G) * (8 * G);
  constexpr int kSlices = sizeof(R) == 8 ? 4 : 1;   // of 8 terms added before the accumulators take them
  R* Xj = diag ? X : X + KS * pitch;
  const int nload_i = KS * ri, nload = diag ? nload_i : nload_i + KS * rj;
  __syncthreads();                            // roff
  // this thread's elements of a slab: row offset, index of the slab and place in X (packed); rows past the
  // tile read its first row and are zeroed by the mask
  uint32_t erow[kGLoad];
  int eat[kGLoad];
  unsigned emask = 0;
#pragma unroll
  for (int i = 0; i < kGLoad; ++i) {
    int e = tid + i * kGThreads;
    const bool in = e < nload;
    const int side = in && e >= nload_i;
    if (side) e -= nload_i;
    const int nr4 = (side ? rj : ri) / 4, h = e >> 5, kh = h / nr4;
    const int r = (h - kh * nr4) * 4 + ((e >> 3) & 3), kk = kh * 8 + (e & 7);
    const bool live = in && r < (side ? nj : ni);
    erow[i] = live ? roff[side][r] : 0u;
    eat[i] = in ? ((kk << 16) | (side * KS * pitch + kk * pitch + r)) : -1;
    emask |= live ? 1u << i : 0u;
  }

  using Pair = typename std::conditional<sizeof(R) == 8, double, float>::type;
  Pair acc[4][4], accl[4][4];     // accl: low parts of the float pairs (unused for FP64)
  R part[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = accl[a][b] = part[a][b] = 0;
  auto flush = [&]() {
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) {
        if constexpr (sizeof(R) == 8) acc[a][b] += part[a][b];
        else two_sum_acc(acc[a][b], accl[a][b], part[a][b]);
        part[a][b] = 0;
      }
  };
  uint32_t rmask[8];
#pragma unroll
  for (int d = 0; d < 8; ++d) rmask[d] = d < jb.nrest ? gram_mask(jobs, bidx, jb.rdir[d]) : 0u;
  uint32_t unit = 0;                          // charge of the summed legs of one value
#pragma unroll
  for (int n = 0; n < 4; ++n)
    if ((jb.unit >> n) & 1u) unit ^= gram_mask(jobs, bidx, n);

  for (int64_t kb = k0; kb < k1; kb += kGList) {
    // offsets of the indices of charge q among the next kGList, in increasing order (K <= 16^6 < 2^32: 32-bit
    // decoding, division by a bond dimension as a multiplication by its rounded-up reciprocal)
    uint32_t off[8];
    unsigned keep[8];
    constexpr int kIter = (kGList + kGThreads - 1) / kGThreads;
    static_assert(kIter <= 8, "decode rounds");
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kIter; ++it) {
      const int64_t k = kb + it * kGThreads + tid;
      bool in = it * kGThreads + tid < kGList && k < k1;
      uint32_t r = (uint32_t)k, o = 0, c = unit;
#pragma unroll
      for (int d = 7; d >= 0; --d) {
        if (d < jb.nrest) {
          const uint32_t n = (uint32_t)jb.rdims[d];
          const uint32_t hi = __umulhi(r, jb.rmagic[d]);
          const uint32_t i = r - hi * n;
          r = hi;
          o += i * (uint32_t)jb.rst[d];
          c ^= rmask[d] >> i;
        }
      }
      in = in && (int)(c & 1u) == q;
      off[it] = o;
      keep[it] = __ballot_sync(0xffffffffu, in);
      if (lane == 0) wcnt[it * (kGThreads / 32) + (tid >> 5)] = __popc(keep[it]);
    }
    __syncthreads();
    if (tid < 32) {                           // exclusive prefix of the counts, three per lane
      static_assert(kIter * (kGThreads / 32) <= 96, "one warp scans the counts");
      int c[3], t = 0;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        c[i] = lane * 3 + i < kIter * (kGThreads / 32) ? wcnt[lane * 3 + i] : 0;
        t += c[i];
      }
      int s = t;
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, s, o);
        if (lane >= o) s += u;
      }
      if (lane == 31) wcnt[8 * (kGThreads / 32)] = s;
      s -= t;
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (lane * 3 + i < kIter * (kGThreads / 32)) wcnt[lane * 3 + i] = s;
        s += c[i];
      }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kIter; ++it)
      if ((keep[it] >> lane) & 1u)
        list[wcnt[it * (kGThreads / 32) + (tid >> 5)] + __popc(keep[it] & ((1u << lane) - 1u))] = off[it];
    __syncthreads();
    const int nk = wcnt[8 * (kGThreads / 32)];
    R reg[kGLoad];
    auto load = [&](int ks) {
#pragma unroll
      for (int i = 0; i < kGLoad; ++i) {
        const int k = ks + (eat[i] >> 16);
        reg[i] = ((emask >> i) & 1u) && k < nk ? T[erow[i] + list[k]] : (R)0;
      }
    };
    auto term = [&](int kk) {
      R vi[4], vj[4];
      const R* xi = X + kk * pitch + bi * 4;
      const R* xj = Xj + kk * pitch + bj * 4;
      if constexpr (sizeof(R) == 4) {
        const float4 u = *(const float4*)xi, w = *(const float4*)xj;
        vi[0] = u.x, vi[1] = u.y, vi[2] = u.z, vi[3] = u.w;
        vj[0] = w.x, vj[1] = w.y, vj[2] = w.z, vj[3] = w.w;
      } else {
        const double2 u0 = *(const double2*)xi, u1 = *(const double2*)(xi + 2);
        const double2 w0 = *(const double2*)xj, w1 = *(const double2*)(xj + 2);
        vi[0] = u0.x, vi[1] = u0.y, vi[2] = u1.x, vi[3] = u1.y;
        vj[0] = w0.x, vj[1] = w0.y, vj[2] = w1.x, vj[3] = w1.y;
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) part[a][b] = fma(vi[a], vj[b], part[a][b]);
    };
    int terms = 0;                            // slices (whole) or terms since the last flush
    load(0);
    for (int ks = 0; ks < nk; ks += KS) {
#pragma unroll
      for (int i = 0; i < kGLoad; ++i)
        if (eat[i] >= 0) X[eat[i] & 0xffff] = reg[i];
      __syncthreads();
      if (ks + KS < nk) load(ks + KS);
      if (works) {
        if (whole) {
          for (int kk = g; kk < KS; kk += 8 * G) {
#pragma unroll
            for (int u = 0; u < 8; ++u) term(kk + u * G);
            if (++terms == kSlices) {
              flush();
              terms = 0;
            }
          }
        } else {
          for (int kk = g; kk < KS; kk += G) {
            term(kk);
            if (++terms == 8 * kSlices) {
              flush();
              terms = 0;
            }
          }
        }
      }
      __syncthreads();
    }
    if (works) flush();
  }
  // the groups' sums, added pairwise (groups h .. 2 h - 1 onto 0 .. h - 1): FP64, or pairs of floats
  {
    Pair* red = (Pair*)X;                     // at most 144 groups x blocks, 16 entries (and low parts): 18 KB
    for (int n = G; n > 1;) {
      const int h = (n + 1) / 2;
      __syncthreads();
      if (g >= h && g < n)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int o = e * (n - h) * nblk + tid - h * nblk;
          red[o] = acc[e / 4][e % 4];
          if constexpr (sizeof(R) == 4) red[16 * (n - h) * nblk + o] = accl[e / 4][e % 4];
        }
      __syncthreads();
      if (g < n - h)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int o = e * (n - h) * nblk + tid;
          if constexpr (sizeof(R) == 8) {
            acc[e / 4][e % 4] += red[o];
          } else {
            two_sum_acc(acc[e / 4][e % 4], accl[e / 4][e % 4], red[o]);
            accl[e / 4][e % 4] += red[16 * (n - h) * nblk + o];
          }
        }
      n = h;
    }
  }
  if (g != 0) return;
  double* out = jb.partial + bidx * jobs.sPart + (int64_t)blockIdx.x * Rn * Rn;
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    const int i = bi * 4 + a;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = bj * 4 + b;
      if (i >= ni || j >= nj) continue;
      const int oi = rout[0][i], oj = rout[1][j];
      const double v = (double)acc[a][b] + (double)accl[a][b];
      out[oi * Rn + oj] = v;
      if (!diag || bi != bj) out[oj * Rn + oi] = v;   // the mirrored entry (a diagonal block has both itself)
    }
  }
}

template <typename R>
cudaError_t launch_gram(const GramPack& jobs, int njobs, int Rmax, int nchunks, cudaStream_t st) {
  GramPack p = jobs;
  for (int i = 0; i < njobs; ++i) {
    // summed legs of one value leave, but for their charge (unit); reciprocals ceil(2^32 / n) of the others (exact
    // quotients below 2^28)
    GramJob& j = p.j[i];
    int n = 0;
    j.unit = 0;
    for (int d = 0; d < j.nrest; ++d) {
      if (j.rdims[d] == 1) {
        j.unit ^= 1u << j.rdir[d];
        continue;
      }
      j.rdims[n] = j.rdims[d];
      j.rst[n] = j.rst[d];
      j.rdir[n] = j.rdir[d];
      j.rmagic[n] = (uint32_t)(((1ull << 32) + j.rdims[n] - 1) / j.rdims[n]);
      ++n;
    }
    j.nrest = n;
  }
  // tile pairs of both charges: at most those of one charge of all rows, and one more tile
  const int nt = (Rmax + kGT - 1) / kGT + (jobs.sectors ? 1 : 0);
  dim3 grid(nchunks, nt * (nt + 1) / 2, njobs * jobs.batch);
  gram_kernel<R><<<grid, kGramThreads<R>, 0, st>>>(p, njobs, nchunks);
  return cudaGetLastError();
}
template cudaError_t launch_gram<double>(const GramPack&, int, int, int, cudaStream_t);
template cudaError_t launch_gram<float>(const GramPack&, int, int, int, cudaStream_t);

// out_i[e] = sum_c partial_i[c][e] for every job i of the pack (and batch element), in one
// launch; job i of element b goes to out[(b njobs + i) out_stride]. A block takes 32
// consecutive entries of one job; its 8 warps add interleaved chunk subsets (warp w: chunks
// c = w mod 8, in increasing c) and the 8 warp sums are added in warp order, so the result
// does not depend on scheduling.
__global__ void __launch_bounds__(256) gram_reduce_kernel(const __grid_constant__ GramPack jobs, int njobs,
                                                          int nchunks, int64_t out_stride, double* __restrict__ out) {
  const int bidx = blockIdx.y / njobs;
  const GramJob& jb = jobs.j[blockIdx.y - bidx * njobs];
  const double* partial = jb.partial + bidx * jobs.sPart;
  const int Rn = jb.D1 * jb.D2;
  const int64_t RR = (int64_t)Rn * Rn;
  const uint32_t m1 = gram_mask(jobs, bidx, jb.dir1), m2 = gram_mask(jobs, bidx, jb.dir2);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __shared__ double red[8][32];
  for (int64_t e0 = (int64_t)blockIdx.x * 32; e0 < RR; e0 += (int64_t)gridDim.x * 32) {
    const int64_t e = e0 + lane;
    double s = 0;
    // entries between charges are exact zeros that no chunk wrote
    bool in = e < RR;
    if (in) {
      const int i = (int)(e / Rn), j = (int)(e - (int64_t)i * Rn);
      const uint32_t c = (m1 >> (i / jb.D2)) ^ (m2 >> (i % jb.D2)) ^ (m1 >> (j / jb.D2)) ^ (m2 >> (j % jb.D2));
      in = !(c & 1u);
    }
    if (in)
      for (int c = w; c < nchunks; c += 8) s += partial[(int64_t)c * RR + e];
    red[w][lane] = s;
    __syncthreads();
    if (w == 0 && e < RR) {
      double t = 0;
      for (int q = 0; q < 8; ++q) t += red[q][lane];
      out[(int64_t)blockIdx.y * out_stride + e] = t;
    }
    __syncthreads();
  }
}

cudaError_t launch_gram_reduce(const GramPack& jobs, int njobs, int nchunks, int64_t RRmax, int64_t out_stride,
                               double* out, cudaStream_t st) {
  int64_t blocks = (RRmax + 31) / 32;
  if (blocks > 1024) blocks = 1024;
  gram_reduce_kernel<<<dim3((unsigned)blocks, (unsigned)(njobs * jobs.batch)), 256, 0, st>>>(jobs, njobs, nchunks,
                                                                                             out_stride, out);
  return cudaGetLastError();
}

// G[(a1 a2),(b1 b2)] = sum_{k,k'} A1[(a1,k),(b1,k')] A2[(a2,k),(b2,k')], FP64.
// blockIdx.y: the matrix, its halves at half[2 y RRs] and half[(2 y + 1) RRs].
__global__ void gram_merge_kernel(const double* __restrict__ half, int64_t RRs, int Dn, int Dk, double* __restrict__ G,
                                  int64_t nn) {
  const double* A1 = half + 2 * blockIdx.y * RRs;
  const double* A2 = A1 + RRs;
  G += blockIdx.y * nn;
  const int n = Dn * Dn;
  const int Rk = Dn * Dk;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int row = e / n, col = e % n;
    const int a1 = row / Dn, a2 = row % Dn, b1 = col / Dn, b2 = col % Dn;
    double s = 0;
    for (int k = 0; k < Dk; ++k)
      for (int kp = 0; kp < Dk; ++kp)
        s = fma(A1[(int64_t)(a1 * Dk + k) * Rk + b1 * Dk + kp], A2[(int64_t)(a2 * Dk + k) * Rk + b2 * Dk + kp], s);
    G[e] = s;
  }
}

cudaError_t launch_gram_merge(const double* half, int64_t RRs, int Dn, int Dk, double* G, int64_t nn, int count,
                              cudaStream_t st) {
  const int n2 = Dn * Dn * Dn * Dn;
  gram_merge_kernel<<<dim3((n2 + 127) / 128, count), 128, 0, st>>>(half, RRs, Dn, Dk, G, nn);
  return cudaGetLastError();
}

// One launch for the six Gram matrices of every batch element: blockIdx.y = b * 6 + i * 2 +
// side (same arithmetic and order as gram_merge_kernel).
__global__ void gram_merge_batch_kernel(const double* __restrict__ half, int64_t RRs, int Dn0, int Dn1, int Dn2,
                                        int Dk, double* __restrict__ G, int64_t nn) {
  const int q = blockIdx.y % 6, bidx = blockIdx.y / 6;
  const int i = q / 2;
  const int Dn = i == 0 ? Dn0 : (i == 1 ? Dn1 : Dn2);
  const double* A1 = half + ((int64_t)bidx * 12 + q * 2) * RRs;
  const double* A2 = A1 + RRs;
  double* Gq = G + ((int64_t)bidx * 6 + q) * nn;
  const int n = Dn * Dn;
  const int Rk = Dn * Dk;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n * n; e += gridDim.x * blockDim.x) {
    const int row = e / n, col = e % n;
    const int a1 = row / Dn, a2 = row % Dn, b1 = col / Dn, b2 = col % Dn;
    double s = 0;
    for (int k = 0; k < Dk; ++k)
      for (int kp = 0; kp < Dk; ++kp)
        s = fma(A1[(int64_t)(a1 * Dk + k) * Rk + b1 * Dk + kp], A2[(int64_t)(a2 * Dk + k) * Rk + b2 * Dk + kp], s);
    Gq[e] = s;
  }
}

cudaError_t launch_gram_merge_batch(const double* half, int64_t RRs, const int Dn[3], int Dk, double* G, int64_t nn,
                                    int batch, cudaStream_t st) {
  int nmax = 0;
  for (int i = 0; i < 3; ++i) nmax = nmax > Dn[i] * Dn[i] ? nmax : Dn[i] * Dn[i];
  const int blocks = (nmax * nmax + 255) / 256;
  gram_merge_batch_kernel<<<dim3(blocks, 6 * batch), 256, 0, st>>>(half, RRs, Dn[0], Dn[1], Dn[2], Dk, G, nn);
  return cudaGetLastError();
}

}  // namespace hotrg
