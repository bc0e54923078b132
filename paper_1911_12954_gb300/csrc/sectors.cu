// sectors.cu - the block-spin contraction of tensors that conserve the Z2 charge.
//
// Without a field the Ising site tensor has T[i1 .. i8] = 0 exactly when the sum of its
// indices is odd, and every later stage keeps such zeros: the Gram matrices split by the charge
// of the fused index, so do the eigenvectors (the Jacobi tournament never leaves a connected
// component and the canonical gauge projects within a charge), and products of exact zeros are
// exact zeros. Every bond index therefore carries a charge q in {0, 1}: the charge of the
// isometry column it came from. A GEMM operand row (X, Y, c, c', mu) of charge r is nonzero only
// at summed indices (a2, b2, a1', b1', k) of charge r + p (p the tensor's own parity: 0 for T and
// M, 1 for S), and C = A B^T has only the blocks with q(row) + q(column) = the output's parity:
// a quarter of the multiply-adds of the dense product, half of the operand and C bytes.
//
// The sizes of the sectors are known on the device only (they follow from the order of the
// eigenvalues), so nothing here depends on them on the host: sector_tables_kernel ranks the
// rows, the summed indices and the row groups within their charge, and every later kernel of the
// step reads its extents from the SectorPlan. Rows are stored charge 0 first, each row's
// nonzero summed indices packed to the front of its K panels (zero filled up to a k-block), so
// the buffers, the tensor maps and the GEMM pipelines are those of the dense product.
// An isometry column that mixes charges (which exact arithmetic excludes) drops the element to
// "every charge 0" (SectorState::dropped): one sector, the dense product.
//
// Sums run over the nonzero terms in the order of the dense passes, so operands, C entries
// given the same k order, and closed tensors are bit-identical to the dense passes'.
#include "common.cuh"
#include "ttm_device.cuh"

namespace hotrg {

namespace {

__device__ __forceinline__ int bit(uint32_t m, int i) { return (int)(m >> i) & 1; }
// indices below j with charge 1
__device__ __forceinline__ int odd_below(uint32_t m, int j) { return __popc(m & ((1u << j) - 1u)); }

// Rank of the multi-index idx among those of its own charge, in lexicographic order, and that
// charge in the top bit. With N_i(s) the number of index suffixes after leg i of charge s,
// rank = sum_i #{j < idx_i, q(j) = 0} N_i(s_i) + #{j < idx_i, q(j) = 1} N_i(s_i + 1), s_i the
// charge left for the legs from i on.
template <int L>
__device__ __forceinline__ uint32_t sector_rank(const int (&d)[L], const uint32_t (&m)[L], const int (&idx)[L]) {
  int q = 0;
#pragma unroll
  for (int i = 0; i < L; ++i) q ^= bit(m[i], idx[i]);
  int rank = 0, prod = 1, diff = 1, s = 0;   // suffix product of sizes and of (even - odd)
#pragma unroll
  for (int i = L - 1; i >= 0; --i) {
    s ^= bit(m[i], idx[i]);                  // charge of the legs from i on
    const int n1 = odd_below(m[i], idx[i]), n0 = idx[i] - n1;
    const int even = (prod + diff) / 2, odd = (prod - diff) / 2;
    rank += s ? n0 * odd + n1 * even : n0 * even + n1 * odd;
    prod *= d[i];
    diff *= d[i] - 2 * odd_below(m[i], d[i]);
  }
  return (uint32_t)rank | ((uint32_t)q << 31);
}

template <int L>
__device__ __forceinline__ void decode(const int (&d)[L], uint32_t e, int (&idx)[L]) {
#pragma unroll
  for (int i = L - 1; i >= 0; --i) {
    idx[i] = (int)(e % (uint32_t)d[i]);
    e /= (uint32_t)d[i];
  }
}

// multi-indices of charge 0 over L legs
template <int L>
__device__ __forceinline__ int even_count(const int (&d)[L], const uint32_t (&m)[L], int first) {
  int prod = 1, diff = 1;
  for (int i = first; i < L; ++i) {
    prod *= d[i];
    diff *= d[i] - 2 * odd_below(m[i], d[i]);
  }
  return (prod + diff) / 2;
}

}  // namespace

// One thread per table entry; blockIdx.y = element of the group.
__global__ void __launch_bounds__(256) sector_tables_kernel(SectorArgs a) {
  const int e = blockIdx.y;
  const SectorState st = a.state[e];
  const uint32_t* qo = st.charge[a.cur];
  const uint32_t* qn = st.charge[1 - a.cur];
  const uint32_t keep = st.dropped ? 0u : 0xffffffffu;
  const uint32_t ma = qo[a.a] & keep, mb = qo[a.b] & keep, mc = qo[a.c] & keep, mm = qo[a.mu] & keep;
  const uint32_t na = qn[a.a] & keep, nb = qn[a.b] & keep, nc = qn[a.c] & keep;
  const int rd[5] = {a.ca, a.cb, a.Dc, a.Dc, a.Dm};
  const uint32_t rm[5] = {na, nb, mc, mc, mm};
  const int kd[5] = {a.Da, a.Db, a.Da, a.Db, a.Dm};
  const uint32_t km[5] = {ma, mb, ma, mb, mm};
  const int gd[4] = {a.ca, a.cb, a.Dc, a.Dm};
  const uint32_t gm[4] = {na, nb, mc, mm};
  const int rows = a.ca * a.cb * a.Dc * a.Dc * a.Dm, K = a.Da * a.Da * a.Db * a.Db * a.Dm;
  const int groups = a.ca * a.cb * a.Dc * a.Dm;
  SectorTables t = a.tab.at(e);
  const int K0 = even_count(kd, km, 0), G0 = even_count(gd, gm, 0);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows + K + groups; i += gridDim.x * blockDim.x) {
    if (i < rows) {
      int idx[5];
      decode(rd, (uint32_t)i, idx);
      t.row[i] = sector_rank(rd, rm, idx);
    } else if (i < rows + K) {
      int idx[5];
      decode(kd, (uint32_t)(i - rows), idx);
      const uint32_t r = sector_rank(kd, km, idx);
      const int pos = (int)(r & 0x7fffffffu) + ((r >> 31) ? K0 : 0);
      // offsets inside one (X, contracted leg, c, c', mu) block of the first pass's output
      const uint32_t oa = (uint32_t)(idx[0] * a.kA[0] + idx[2] * a.kA[2] + idx[3] * a.kA[3] + idx[4] * a.kA[4]);
      const uint32_t ob = (uint32_t)(idx[0] * a.kB[0] + idx[1] * a.kB[1] + idx[2] * a.kB[2] + idx[4] * a.kB[4]);
      t.kA[pos] = make_uint2(oa, (uint32_t)idx[1]);
      t.kB[pos] = make_uint2(ob, (uint32_t)idx[3]);
    } else {
      const int g = i - rows - K;
      int idx[4];
      decode(gd, (uint32_t)g, idx);
      const uint32_t r = sector_rank(gd, gm, idx);
      t.grank[g] = r;
      t.grp[(int)(r & 0x7fffffffu) + ((r >> 31) ? G0 : 0)] = (uint32_t)g;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    SectorPlan& p = *t.plan;
    const int r0 = even_count(rd, rm, 1), r1 = rows / a.ca - r0;   // rows of one X by the other legs' charge
    const int g0 = even_count(gd, gm, 1), g1 = groups / a.ca - g0;
    p.row[0][0] = p.row[1][0] = p.grp[0][0] = p.grp[1][0] = 0;
    for (int x = 0; x < a.ca; ++x) {
      const int q = bit(na, x);
      p.row[0][x + 1] = p.row[0][x] + (q ? r1 : r0);
      p.row[1][x + 1] = p.row[1][x] + (q ? r0 : r1);
      p.grp[0][x + 1] = p.grp[0][x] + (q ? g1 : g0);
      p.grp[1][x + 1] = p.grp[1][x] + (q ? g0 : g1);
    }
    p.K[0] = K0;
    p.K[1] = K - K0;
    p.na = na;
    p.nb = nb;
    p.nc = nc;
    p.mb = mb;
    p.mc = mc;
    p.mm = mm;
  }
}

// Largest dynamic shared memory of the kernels below (bond dimension 16 in FP64: 80 KB); set once
// per device ahead of any launch, so no launch inside a stream capture does host-side set-up.
constexpr int kSectorSmem = 96 * 1024;

cudaError_t launch_sector_tables(const SectorArgs& a, int ne, cudaStream_t st) {
  const int64_t n = (int64_t)a.ca * a.cb * a.Dc * a.Dc * a.Dm + (int64_t)a.Da * a.Da * a.Db * a.Db * a.Dm +
                    (int64_t)a.ca * a.cb * a.Dc * a.Dm;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  sector_tables_kernel<<<dim3((unsigned)blocks, ne), 256, 0, st>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------- operands
// Second half-contraction pass: operand[row(X, Y, c, c', mu), k] = sum_j U[j, r, Y] O1[X, j, c, c', mu, rest(k)]
// with k = (r, rest) (r: the new leg b2 of A, b1' of B; j: the contracted leg). A block takes one
// (X, c, c', mu) and one charge Q of k; its threads walk the packed summed indices two at a time, so
// stores of a warp are contiguous, and each thread sums only the j whose charge fits. The Y of one
// charge (the only nonzero rows) are produced four at a time.
template <int MODE, typename R>
__device__ __forceinline__ void sector_store2(R* out, R* out_lo, int64_t o, R v0, R v1) {
  if constexpr (MODE == kTTMSplitF16) {
    const float f0 = (float)v0, f1 = (float)v1;
    const __half h0 = __float2half_rn(f0), h1 = __float2half_rn(f1);
    *(__half2*)((__half*)out + o) = __halves2half2(h0, h1);
    *(__half2*)((__half*)out_lo + o) =
        __halves2half2(__float2half_rn(f0 - __half2float(h0)), __float2half_rn(f1 - __half2float(h1)));
  } else if constexpr (MODE == kTTMSplitTF32) {
    const float f0 = (float)v0, f1 = (float)v1;
    const float h0 = tf32_round(f0), h1 = tf32_round(f1);
    *(float2*)((float*)out + o) = make_float2(h0, h1);
    *(float2*)((float*)out_lo + o) = make_float2(tf32_round(f0 - h0), tf32_round(f1 - h1));
  } else if constexpr (MODE == kTTMSplitOz) {
    oz_store2((__half*)out, (__half*)out_lo - (__half*)out, o, (double)v0, (double)v1);
  } else {
    out[o] = v0;
    out[o + 1] = v1;
  }
}

template <typename R, int MODE>
__global__ void __launch_bounds__(256) sector_operand_kernel(const R* __restrict__ in, const R* __restrict__ U,
                                                             R* __restrict__ out, R* __restrict__ out_lo,
                                                             const __grid_constant__ SectorOperand a) {
  const int e = blockIdx.y, Q = blockIdx.z;
  const SectorTables t = a.tab.at(e);
  const SectorPlan& p = *t.plan;
  in += e * a.in_bs;
  U += e * a.u_bs;
  out = elem_out<R, MODE>(out, e * a.out_bs);
  out_lo = elem_out<R, MODE>(out_lo, e * a.out_bs);
  unsigned* amax = a.amax ? a.amax + e * a.amax_bs : nullptr;
  const R uscale = (R)split_scale<MODE>(amax);
  extern __shared__ __align__(16) unsigned char fsm[];
  R* Us = (R*)fsm;                      // [2][Db][Db][Yp]: (charge of Y, j, r, slot of Y), zero past the last slot
  __shared__ int ny[2], nj[2], ylist[2][kMaxLeg], jlist[2][kMaxLeg];
  const int Db = a.Db, Yp = (a.cb + 3) / 4 * 4;
  const uint32_t mb = p.mb, nb = p.nb, na = p.na, mc = p.mc, mm = p.mm;
  if (threadIdx.x < 2) {
    const int q = threadIdx.x;
    int n = 0;
    for (int y = 0; y < a.cb; ++y)
      if (bit(nb, y) == q) ylist[q][n++] = y;
    ny[q] = n;
    n = 0;
    for (int j = 0; j < Db; ++j)
      if (bit(mb, j) == q) jlist[q][n++] = j;
    nj[q] = n;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * Db * Db * Yp; i += blockDim.x) {
    const int sl = i % Yp, r = (i / Yp) % Db, j = (i / (Yp * Db)) % Db, q = i / (Yp * Db * Db);
    Us[i] = sl < ny[q] ? U[j * a.u_j + r * a.u_r + ylist[q][sl]] * uscale : (R)0;
  }
  __syncthreads();
  const int KQ = p.K[Q], Kpad = (KQ + a.kalign - 1) / a.kalign * a.kalign;
  const uint2* kt = (a.sideB ? t.kB : t.kA) + (Q ? p.K[0] : 0);
  const int rows0 = p.row[0][a.x0 + a.xs] - p.row[0][a.x0];   // charge-0 rows of the slice
  const int rq = Q ^ a.parity;                                // charge of the rows with nonzero entries
  const int rbase = (rq ? rows0 : 0) - p.row[rq][a.x0];
  R tmax = 0;
  for (int o = blockIdx.x; o < a.nouter; o += gridDim.x) {
    int r = o;
    const int m = r % a.Dm;
    r /= a.Dm;
    const int c1 = r % a.Dc;
    r /= a.Dc;
    const int c0 = r % a.Dc;
    const int X = r / a.Dc;
    const int y = rq ^ bit(na, a.x0 + X) ^ bit(mc, c0) ^ bit(mc, c1) ^ bit(mm, m);
    const R* src = in + X * a.in_x + c0 * a.in_c0 + c1 * a.in_c1 + m * a.in_m;
    const uint32_t* rt = t.row + (((int64_t)(a.x0 + X) * a.cb * a.Dc + c0) * a.Dc + c1) * a.Dm + m;
    const int64_t ystep = (int64_t)a.Dc * a.Dc * a.Dm;
    const int nyy = ny[y];
    const R* Uy = Us + (size_t)y * Db * Db * Yp;
    for (int k = 2 * threadIdx.x; k < Kpad; k += 2 * blockDim.x) {
      const int pn = a.P > 1 ? k / a.kps : 0;
      const int64_t ocol = (int64_t)pn * a.rows * a.kps + (k - pn * a.kps);
      for (int yb = 0; yb < nyy; yb += 4) {
        R v[2][4];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
#pragma unroll
          for (int s = 0; s < 4; ++s) v[h][s] = 0;
          if (k + h < KQ) {
            const uint2 q = kt[k + h];
            const R* x = src + q.x;
            const int jc = y ^ bit(mb, (int)q.y);   // U[j, r, Y] is nonzero for q(j) + q(r) = q(Y)
            const int n = nj[jc];
            const R* u = Uy + (size_t)q.y * Yp + yb;
#pragma unroll 4
            for (int i = 0; i < n; ++i) {
              const int j = jlist[jc][i];
              const R xv = x[(int64_t)j * a.in_j];
              const R* uj = u + (size_t)j * Db * Yp;
#pragma unroll
              for (int s = 0; s < 4; ++s) v[h][s] = fma(uj[s], xv, v[h][s]);
            }
          }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          if (yb + s >= nyy) break;
          if (MODE == kTTMMaxAbs) {
            tmax = fmax(tmax, fmax(fabs(v[0][s]), fabs(v[1][s])));
          } else {
            const int row = (int)(rt[ylist[y][yb + s] * ystep] & 0x7fffffffu) + rbase;
            sector_store2<MODE>(out, out_lo, (int64_t)row * a.kps + ocol, v[0][s], v[1][s]);
          }
        }
      }
    }
  }
  if (MODE == kTTMMaxAbs) merge_max(amax, (double)tmax, a.amax_mul);   // every thread gets here
}

template <typename R>
cudaError_t launch_sector_operand(const R* in, const R* U, R* out, R* out_lo, const SectorOperand& a, int ne, int mode,
                                  cudaStream_t st) {
  const int Yp = (a.cb + 3) / 4 * 4;
  const size_t smem = (size_t)2 * a.Db * a.Db * Yp * sizeof(R);
  if (smem > (size_t)kSectorSmem) return cudaErrorInvalidValue;
  int64_t bx = a.nouter;
  const int64_t cap = 152 * 32 / ne > 64 ? 152 * 32 / ne : 64;
  if (bx > cap) bx = cap;
  const dim3 g((unsigned)bx, ne, 2);
  auto go = [&](auto kernel) -> cudaError_t {
    kernel<<<g, 256, smem, st>>>(in, U, out, out_lo, a);
    return cudaGetLastError();
  };
  switch (mode) {
    case kTTMStore: return go(sector_operand_kernel<R, kTTMStore>);
    case kTTMMaxAbs: return go(sector_operand_kernel<R, kTTMMaxAbs>);
    case kTTMSplitF16: if constexpr (sizeof(R) == 4) return go(sector_operand_kernel<R, kTTMSplitF16>); break;
    case kTTMSplitTF32: if constexpr (sizeof(R) == 4) return go(sector_operand_kernel<R, kTTMSplitTF32>); break;
    case kTTMSplitOz: if constexpr (sizeof(R) == 8) return go(sector_operand_kernel<R, kTTMSplitOz>); break;
  }
  return cudaErrorInvalidValue;
}
template cudaError_t launch_sector_operand<float>(const float*, const float*, float*, float*, const SectorOperand&, int,
                                                  int, cudaStream_t);
template cudaError_t launch_sector_operand<double>(const double*, const double*, double*, double*,
                                                   const SectorOperand&, int, int, cudaStream_t);

// ---------------------------------------------------------------------------- closing passes
// First closing pass: O3[Z][m][n] = sum_{c1, c2} U[c1, c2, Z] C[row(X, Y, c1, c1', mu1)][col(X', Y', c2, c2', mu2')]
// with m, n the ranked row groups (X, Y, c1', mu1) and (X', Y', c2', mu2'). A block takes 256 column
// groups of one charge t and row groups of one charge r, four at a time: only the pairs (c1, c2) with
// q(c1) + q(c2) = s (s = r + t + the output's parity) and the Z of charge s are nonzero, the same for
// the whole block, so no lane is idle; the entries of the other Z are neither written nor read.
template <typename R, int NZ>
__global__ void __launch_bounds__(256) sector_close1_kernel(const R* __restrict__ C, const R* __restrict__ U,
                                                            R* __restrict__ O3,
                                                            const __grid_constant__ SectorClose a) {
  constexpr int RG = 4;
  const int e = blockIdx.z;
  const SectorTables t = a.tab.at(e);
  const SectorPlan& p = *t.plan;
  C += e * a.c_bs;
  U += e * a.u_bs;
  O3 += e * a.o3_bs;
  const int Dc = a.Dc, tid = threadIdx.x;
  const int g0 = p.grp[0][a.x20], n0 = p.grp[0][a.x20 + a.xs2] - g0;
  const int g1 = p.grp[1][a.x20], n1 = p.grp[1][a.x20 + a.xs2] - g1;
  const int ch0 = (n0 + 255) / 256;
  const int tq = (int)blockIdx.x < ch0 ? 0 : 1;                 // charge of the column groups
  const int i0 = (tq ? (int)blockIdx.x - ch0 : (int)blockIdx.x) * 256;
  const int ncol = tq ? n1 : n0;
  if (i0 >= ncol) return;
  extern __shared__ __align__(16) unsigned char fsm[];
  R* Us = (R*)fsm;                                   // [2][Dc][Dc][NZ]: (charge of Z, c1, c2, slot), zero past the last slot
  int* rks = (int*)(Us + (size_t)2 * Dc * Dc * NZ);  // [Dc][256] column of c2
  __shared__ int nz[2], nc[2], zlist[2][kMaxLeg], clist[2][kMaxLeg];
  if (tid < 2) {
    int n = 0;
    for (int z = 0; z < a.cc; ++z)
      if (bit(p.nc, z) == tid) zlist[tid][n++] = z;
    nz[tid] = n;
    n = 0;
    for (int c = 0; c < Dc; ++c)
      if (bit(p.mc, c) == tid) clist[tid][n++] = c;
    nc[tid] = n;
  }
  __syncthreads();
  for (int i = tid; i < 2 * Dc * Dc * NZ; i += 256) {
    const int sl = i % NZ, c2 = (i / NZ) % Dc, c1 = (i / (NZ * Dc)) % Dc, q = i / (NZ * Dc * Dc);
    Us[i] = sl < nz[q] ? U[((int64_t)c1 * Dc + c2) * a.cc + zlist[q][sl]] : (R)0;
  }
  const uint32_t* grp0 = t.grp;                       // ranked groups of charge 0, then of charge 1
  const int G0 = p.grp[0][a.ca];
  const int inner = Dc * a.Dm;                        // (c', mu) extent of a group
  const bool live = i0 + tid < ncol;
  const int gi = live ? i0 + tid : ncol - 1;
  {
    const uint32_t g = grp0[(tq ? G0 + g1 : g0) + gi];
    const uint32_t hi = g / (uint32_t)inner, rem = g - hi * inner;
    for (int c2 = 0; c2 < Dc; ++c2) {
      const uint32_t r = t.row[((int64_t)hi * Dc + c2) * inner + rem];
      rks[c2 * 256 + tid] = (int)(r & 0x7fffffffu) - p.row[r >> 31][a.x20];
    }
  }
  __syncthreads();
  const int rows0 = p.row[0][a.x0 + a.xs] - p.row[0][a.x0];
  const int mg0 = p.grp[0][a.x0 + a.xs] - p.grp[0][a.x0];   // charge-0 row groups of the slice
  const int64_t GR = (int64_t)a.xs * a.cb * inner, GC = (int64_t)a.xs2 * a.cb * inner;
  const int64_t ocol = (tq ? n0 : 0) + gi;
  for (int rq = 0; rq < 2; ++rq) {
    const int gbase = p.grp[rq][a.x0], nrow = p.grp[rq][a.x0 + a.xs] - gbase;
    const int s = rq ^ tq ^ a.parity;
    const int nzs = nz[s];
    if (nzs == 0) continue;
    for (int b = blockIdx.y * RG; b < nrow; b += gridDim.y * RG) {
      uint32_t hi[RG], rem[RG];
#pragma unroll
      for (int i = 0; i < RG; ++i) {
        const uint32_t g = grp0[(rq ? G0 : 0) + gbase + min(b + i, nrow - 1)];
        hi[i] = g / (uint32_t)inner;
        rem[i] = g - hi[i] * inner;
      }
      R acc[RG][NZ];
#pragma unroll
      for (int i = 0; i < RG; ++i)
#pragma unroll
        for (int z = 0; z < NZ; ++z) acc[i][z] = 0;
      for (int c1 = 0; c1 < Dc; ++c1) {
        const int q1 = bit(p.mc, c1), rc = rq ^ q1, jc = s ^ q1;
        const int roff = (rc ? rows0 : 0) - p.row[rc][a.x0];
        const R* cp[RG];
#pragma unroll
        for (int i = 0; i < RG; ++i) {
          const int row = (int)(t.row[((int64_t)hi[i] * Dc + c1) * inner + rem[i]] & 0x7fffffffu) + roff;
          cp[i] = C + (int64_t)row * a.ldc;
        }
        const int n = nc[jc];
        const R* u1 = Us + ((size_t)s * Dc + c1) * Dc * NZ;
        int k = 0;
        for (; k + 4 <= n; k += 4) {
          R x[4][RG];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int col = rks[clist[jc][k + q] * 256 + tid];
#pragma unroll
            for (int i = 0; i < RG; ++i) x[q][i] = cp[i][col];
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const R* u = u1 + clist[jc][k + q] * NZ;
#pragma unroll
            for (int zb = 0; zb < NZ; zb += 4) {
              if (zb < nzs) {
#pragma unroll
                for (int z = 0; z < 4; ++z) {
                  const R w = u[zb + z];
#pragma unroll
                  for (int i = 0; i < RG; ++i) acc[i][zb + z] = fma(w, x[q][i], acc[i][zb + z]);
                }
              }
            }
          }
        }
        for (; k < n; ++k) {
          const int col = rks[clist[jc][k] * 256 + tid];
          R x[RG];
#pragma unroll
          for (int i = 0; i < RG; ++i) x[i] = cp[i][col];
          const R* u = u1 + clist[jc][k] * NZ;
#pragma unroll
          for (int zb = 0; zb < NZ; zb += 4) {
            if (zb < nzs) {
#pragma unroll
              for (int z = 0; z < 4; ++z) {
                const R w = u[zb + z];
#pragma unroll
                for (int i = 0; i < RG; ++i) acc[i][zb + z] = fma(w, x[i], acc[i][zb + z]);
              }
            }
          }
        }
      }
      if (live) {
#pragma unroll
        for (int i = 0; i < RG; ++i) {
          if (b + i >= nrow) break;
          const int64_t orow = (rq ? mg0 : 0) + b + i;
#pragma unroll
          for (int z = 0; z < NZ; ++z)
            if (z < nzs) O3[((int64_t)zlist[s][z] * GR + orow) * GC + ocol] = acc[i][z];
        }
      }
    }
  }
}

// Second closing pass: T'[X, X', Y, Y', Z, Z', mu1, mu2'] = sum_{c1', c2'} U[c1', c2', Z'] O3[Z][m][n], one thread
// per output fibre (every leg but Z') in the output's own leg order; terms of the wrong charge are
// skipped (O3 does not hold them) and the Z' of the wrong charge come out as exact zeros, as U's.
template <typename R, int NZ>
__global__ void __launch_bounds__(256) sector_close2_kernel(const R* __restrict__ O3, const R* __restrict__ U,
                                                            R* __restrict__ T, const __grid_constant__ SectorClose a) {
  const int e = blockIdx.y;
  const SectorTables t = a.tab.at(e);
  const SectorPlan& p = *t.plan;
  O3 += e * a.o3_bs;
  U += e * a.u_bs;
  T += e * a.t_bs;
  const int Dc = a.Dc;
  extern __shared__ __align__(16) unsigned char fsm[];
  R* Us = (R*)fsm;                                   // [Dc][Dc][NZ], zero past cc
  for (int i = threadIdx.x; i < Dc * Dc * NZ; i += blockDim.x) {
    const int z = i % NZ;
    Us[i] = z < a.cc ? U[(int64_t)(i / NZ) * a.cc + z] : (R)0;
  }
  __syncthreads();
  const int inner = Dc * a.Dm;
  const int64_t GR = (int64_t)a.xs * a.cb * inner, GC = (int64_t)a.xs2 * a.cb * inner;
  const int m0 = p.grp[0][a.x0 + a.xs] - p.grp[0][a.x0], n0 = p.grp[0][a.x20 + a.xs2] - p.grp[0][a.x20];
  const int moff[2] = {-p.grp[0][a.x0], m0 - p.grp[1][a.x0]};
  const int noff[2] = {-p.grp[0][a.x20], n0 - p.grp[1][a.x20]};
  const uint32_t mc = p.mc;
  for (int64_t f = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; f < a.nfib; f += (int64_t)gridDim.x * blockDim.x) {
    uint32_t r = (uint32_t)f;
    int mg = a.x0 * a.cb * inner, ng = a.x20 * a.cb * inner, Z = 0;
    int64_t to = 0;
#pragma unroll
    for (int d = 6; d >= 0; --d) {
      const uint32_t n = (uint32_t)a.fd[d];
      const int i = (int)(r % n);
      r /= n;
      mg += i * a.fm[d];
      ng += i * a.fn[d];
      Z += i * a.fz[d];
      to += i * a.ft[d];
    }
    R acc[NZ];
#pragma unroll
    for (int z = 0; z < NZ; ++z) acc[z] = 0;
    // charge of (c1', c2') that reaches a nonzero entry
    const int qm = (int)(t.grank[mg] >> 31) ^ bit(mc, 0), qn = (int)(t.grank[ng] >> 31) ^ bit(mc, 0);
    const int s = qm ^ qn ^ bit(p.nc, Z) ^ a.parity;
    const R* o3 = O3 + (int64_t)Z * GR * GC;
    for (int c1 = 0; c1 < Dc; ++c1) {
      const uint32_t gr = t.grank[mg + c1 * a.Dm];
      const R* row = o3 + (int64_t)((int)(gr & 0x7fffffffu) + moff[gr >> 31]) * GC;
      const int want = s ^ bit(mc, c1);
      const R* u1 = Us + (size_t)c1 * Dc * NZ;
#pragma unroll 4
      for (int c2 = 0; c2 < Dc; ++c2) {
        R x = 0;
        if (bit(mc, c2) == want) {
          const uint32_t gn = t.grank[ng + c2 * a.Dm];
          x = row[(int)(gn & 0x7fffffffu) + noff[gn >> 31]];
        }
        const R* u = u1 + c2 * NZ;
#pragma unroll
        for (int z = 0; z < NZ; ++z) acc[z] = fma(u[z], x, acc[z]);
      }
    }
#pragma unroll
    for (int z = 0; z < NZ; ++z)
      if (z < a.cc) T[to + z * a.tz] = acc[z];
  }
}

template <typename R>
cudaError_t launch_sector_close(const R* C, const R* U, R* O3, R* T, const SectorClose& a, int ne, cudaStream_t st) {
  if (a.nfib > 0x7fffffffLL || a.nfib < 1) return cudaErrorInvalidValue;
  const int NZ = a.cc <= 4 ? 4 : (a.cc <= 8 ? 8 : 16);
  const size_t s1 = (size_t)2 * a.Dc * a.Dc * NZ * sizeof(R) + (size_t)a.Dc * 256 * sizeof(int);
  const size_t s2 = (size_t)a.Dc * a.Dc * NZ * sizeof(R);
  if (s1 > (size_t)kSectorSmem) return cudaErrorInvalidValue;
  const int64_t cols = (int64_t)a.xs2 * a.cb * a.Dc * a.Dm, rowg = (int64_t)a.xs * a.cb * a.Dc * a.Dm;
  const int64_t bx = (cols + 255) / 256 + 1;
  int64_t by = (152 * 12 + bx * ne - 1) / (bx * ne);
  by = by < 1 ? 1 : by;
  by = by > (rowg + 7) / 8 ? (rowg + 7) / 8 : by;      // four row groups of one charge per step
  const dim3 g1((unsigned)bx, (unsigned)by, ne);
  int64_t b2 = (a.nfib + 255) / 256;
  const int64_t cap = 152 * 16 / ne > 8 ? 152 * 16 / ne : 8;
  if (b2 > cap) b2 = cap;
  const dim3 g2((unsigned)b2, ne);
  auto go = [&](auto k1, auto k2) -> cudaError_t {
    k1<<<g1, 256, s1, st>>>(C, U, O3, a);
    cudaError_t er = cudaGetLastError();
    if (er != cudaSuccess) return er;
    k2<<<g2, 256, s2, st>>>(O3, U, T, a);
    return cudaGetLastError();
  };
  if (NZ == 4) return go(sector_close1_kernel<R, 4>, sector_close2_kernel<R, 4>);
  if (NZ == 8) return go(sector_close1_kernel<R, 8>, sector_close2_kernel<R, 8>);
  return go(sector_close1_kernel<R, 16>, sector_close2_kernel<R, 16>);
}
template cudaError_t launch_sector_close<float>(const float*, const float*, float*, float*, const SectorClose&, int,
                                                cudaStream_t);
template cudaError_t launch_sector_close<double>(const double*, const double*, double*, double*, const SectorClose&, int,
                                                 cudaStream_t);

void sectors_prepare() {
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64 || done[dev]) return;
  done[dev] = true;
  auto set = [](auto k) { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSectorSmem); };
  set(sector_operand_kernel<float, kTTMStore>);
  set(sector_operand_kernel<float, kTTMMaxAbs>);
  set(sector_operand_kernel<float, kTTMSplitF16>);
  set(sector_operand_kernel<float, kTTMSplitTF32>);
  set(sector_operand_kernel<double, kTTMStore>);
  set(sector_operand_kernel<double, kTTMMaxAbs>);
  set(sector_operand_kernel<double, kTTMSplitOz>);
  set(sector_close1_kernel<float, 16>);
  set(sector_close1_kernel<double, 8>);
  set(sector_close1_kernel<double, 16>);
  set(sector_close2_kernel<double, 16>);
  cudaGetLastError();
}

}  // namespace hotrg
