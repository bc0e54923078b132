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
// a quarter of the multiply-adds of the dense product where the charges split evenly (0.29 at D_cut = 8
// near T_c, where 7 of 8 kept columns are even: hotrg_product_share), about half of the operand and C bytes.
//
// The sizes of the sectors are known on the device only (they follow from the order of the
// eigenvalues), so nothing here depends on them on the host: sector_tables_kernel ranks the
// rows, the summed indices and the row groups within their charge, and every later kernel of the
// step reads its extents from the SectorPlan. Rows are stored charge 0 first, each row's
// nonzero summed indices packed to the front of its K panels (zero filled up to a k-block), so
// the buffers, the tensor maps and the GEMM pipelines are those of the dense product.
// An isometry column that mixes charges (which exact arithmetic excludes) drops the element to
// "every charge 0, every parity 0" (SectorState::dropped, SectorPlan::odd): one sector, the dense product.
//
// Operand entries and the closing sums run over their nonzero terms in the dense passes' order. The
// product's summed index comes in the order (b2, b1', a2, a1', k), the dense one's in (a2, b2, a1', b1', k),
// so C agrees with the dense product's up to the order of its sums.
#include <mutex>
#include <type_traits>

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
  const int gd[4] = {a.ca, a.cb, a.Dc, a.Dm};
  const uint32_t gm[4] = {na, nb, mc, mm};
  const int sd[3] = {a.Da, a.Da, a.Dm};
  const uint32_t sm[3] = {ma, ma, mm};
  const int rows = a.ca * a.cb * a.Dc * a.Dc * a.Dm, rests = a.Da * a.Da * a.Dm;
  const int groups = a.ca * a.cb * a.Dc * a.Dm;
  SectorTables t = a.tab.at(e);
  const int S0 = even_count(sd, sm, 0), G0 = even_count(gd, gm, 0);
  const int n0 = (S0 + 1) & ~1, n1 = (rests - S0 + 1) & ~1;   // runs of even length
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rows + rests + groups; i += gridDim.x * blockDim.x) {
    if (i < rows) {
      int idx[5];
      decode(rd, (uint32_t)i, idx);
      t.row[i] = sector_rank(rd, rm, idx);
    } else if (i < rows + rests) {
      // rest (a2, a1', k) of the summed index: offsets in A's (a2, a1', b1', k) and B's (a2, b2, a1', k)
      int idx[3];
      decode(sd, (uint32_t)(i - rows), idx);
      const uint32_t r = sector_rank(sd, sm, idx);
      const int pos = (int)(r & 0x7fffffffu) + ((r >> 31) ? n0 : 0);
      t.kA[pos] = (uint32_t)((idx[0] * a.Da + idx[1]) * a.Db * a.Dm + idx[2]);
      t.kB[pos] = (uint32_t)((idx[0] * a.Db * a.Da + idx[1]) * a.Dm + idx[2]);
    } else {
      const int g = i - rows - rests;
      int idx[4];
      decode(gd, (uint32_t)g, idx);
      const uint32_t r = sector_rank(gd, gm, idx);
      t.grank[g] = r;
      t.grp[(int)(r & 0x7fffffffu) + ((r >> 31) ? G0 : 0)] = (uint32_t)g;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 32) {
    const int k = *a.step;
    if (k < kMaxSteps)
      *(SectorCount*)a.rec[(int64_t)e * kMaxSteps + k].eps[a.mu] =
          SectorCount{even_count(rd, rm, 0), S0, odd_below(mb, a.Db), st.dropped ? 0 : 1};
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
    if (S0 & 1) t.kA[S0] = t.kB[S0] = ~0u;                  // fillers
    if ((rests - S0) & 1) t.kA[n0 + n1 - 1] = t.kB[n0 + n1 - 1] = ~0u;
    p.n3[0] = n0;
    p.n3[1] = n1;
    const int b1 = odd_below(mb, a.Db), b0 = a.Db - b1;
    p.K[0] = (b0 * b0 + b1 * b1) * n0 + 2 * b0 * b1 * n1;
    p.K[1] = (b0 * b0 + b1 * b1) * n1 + 2 * b0 * b1 * n0;
    p.na = na;
    p.nb = nb;
    p.nc = nc;
    p.mb = mb;
    p.mc = mc;
    p.mm = mm;
    p.odd = st.dropped ? 0 : 1;
  }
}

// Largest dynamic shared memory of the kernels below (bond dimension 16 in FP64: 80 KB); set once
// per device ahead of any launch, so no launch inside a stream capture does host-side set-up.
constexpr int kSectorSmem = 96 * 1024;

cudaError_t launch_sector_tables(const SectorArgs& a, int ne, cudaStream_t st) {
  const int64_t n = (int64_t)a.ca * a.cb * a.Dc * a.Dm * (a.Dc + 1) + (int64_t)a.Da * a.Da * a.Dm;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  sector_tables_kernel<<<dim3((unsigned)blocks, ne), 256, 0, st>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------- operands
// Second half-contraction pass: operand[row(X, Y, c, c', mu), k] = sum_j U[j, r, Y] O1[X, j, c, c', mu, rest(k)]
// with j the contracted leg and the summed index k in the order (b2, b1', rest), rest = (a2, a1', k): the new leg
// r is b2 for A and b1' for B, the other of the two is the segment. For fixed (b2, b1') the rests of one charge
// are neighbours in the packed operand (a run, of even length: a filler entry where the count is odd). A block
// takes one (X, c, c', mu); a warp takes 64 rests of one segment and charge, two per lane: their O1 entries are
// nonzero for the j of one charge only, each is loaded once and serves every r and Y, the coefficients are the
// same for the whole warp (broadcast reads from shared memory), and the stores are pairs in runs of 64.
// Instruction issue bounds it (71 % of the issue slots at D_cut = 6, DRAM 26 %), then the writes: at D_cut = 8 a pass
// writes 2.1 GB and reads 0.5 GB (0.4 ms at the copy rate; both sides in one launch 1.67 ms).
template <int MODE, typename R>
__device__ __forceinline__ void sector_store2(R* out, R* out_lo, int64_t o, R v0, R v1) {
  if constexpr (MODE == kTTMSplitF16) {
    const __half2 h = __floats2half2_rn((float)v0, (float)v1);
    const float2 f = __half22float2(h);
    *(__half2*)((__half*)out + o) = h;
    *(__half2*)((__half*)out_lo + o) = __floats2half2_rn((float)v0 - f.x, (float)v1 - f.y);
  } else if constexpr (MODE == kTTMSplitTF32) {
    const float f0 = (float)v0, f1 = (float)v1;
    const float h0 = tf32_round(f0), h1 = tf32_round(f1);
    *(float2*)((float*)out + o) = make_float2(h0, h1);
    *(float2*)((float*)out_lo + o) = make_float2(tf32_round(f0 - h0), tf32_round(f1 - h1));
  } else if constexpr (MODE == kTTMSplitOz) {
    oz_store2((__half*)out, (__half*)out_lo - (__half*)out, o, (double)v0, (double)v1);
  } else if constexpr (sizeof(R) == 8) {
    *(double2*)(out + o) = make_double2(v0, v1);
  } else {
    *(float2*)(out + o) = make_float2(v0, v1);
  }
}

// What the blocks of an operand pass keep in shared memory.
struct OperandShared {
  int ylist[2][kMaxLeg], jlist[2][kMaxLeg];     // Y and j of either charge
  int64_t yrow[2][2][kMaxLeg];                  // row offsets of the Y of either charge, double-buffered
  int base[kMaxLeg][kMaxLeg][2];                // (b2, b1', charge of rest): start of the run
};

// 64 rests (two per lane: x0, x1; live: in the run) times every r and Y, NJ contracted indices.
template <typename R, int MODE, int NJ>
__device__ __forceinline__ void operand_run(const R* x0, const R* x1, bool ok0, bool ok1, bool live, int i, int jc, int sg,
                                            int g, uint32_t mb, int ny0, int ny1, int NJp, int Yp, int buf, const R* Us,
                                            const OperandShared& sh, const SectorOperand& a, R* out, R* out_lo,
                                            unsigned long long& tmax) {
  R xa[NJ > 0 ? NJ : 1], xb[NJ > 0 ? NJ : 1];
#pragma unroll
  for (int j = 0; j < NJ; ++j) {
    const int64_t o = sh.jlist[jc][j] * a.in_j;
    xa[j] = ok0 ? x0[o] : (R)0;
    xb[j] = ok1 ? x1[o] : (R)0;
  }
  const R* uj = Us + (size_t)jc * a.Db * NJp * Yp;
  for (int r = 0; r < a.Db; ++r, uj += (size_t)NJp * Yp) {
    const int y = jc ^ bit(mb, r), nyy = y ? ny1 : ny0;    // U[j, r, Y] is nonzero for q(j) + q(r) = q(Y)
    const int k = (a.sideB ? sh.base[sg][r][g] : sh.base[r][sg][g]) + i;
    const int64_t ocol = k + (int64_t)(a.P > 1 ? k / (int)a.kps : 0) * (a.rows - 1) * a.kps;
    for (int yb = 0; yb < nyy; yb += 4) {
      R va[4] = {0, 0, 0, 0}, vb[4] = {0, 0, 0, 0};
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const R* u = uj + j * Yp + yb;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          va[s] = fma(u[s], xa[j], va[s]);
          vb[s] = fma(u[s], xb[j], vb[s]);
        }
      }
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        if (yb + s >= nyy) break;
        if (MODE == kTTMMaxAbs) {
          // magnitudes as integers (same order): no FP64 comparisons
          if constexpr (sizeof(R) == 8) {
            tmax = max(tmax, (unsigned long long)__double_as_longlong(va[s]) & 0x7fffffffffffffffull);
            tmax = max(tmax, (unsigned long long)__double_as_longlong(vb[s]) & 0x7fffffffffffffffull);
          } else {
            tmax = max(tmax, (unsigned long long)max(__float_as_uint(va[s]) & 0x7fffffffu,
                                                     __float_as_uint(vb[s]) & 0x7fffffffu));
          }
        } else if (live) {
          sector_store2<MODE>(out, out_lo, sh.yrow[buf][y][yb + s] + ocol, va[s], vb[s]);
        }
      }
    }
  }
}

template <typename R, int MODE, int NJM>
__global__ void __launch_bounds__(256) sector_operand_kernel(const __grid_constant__ SectorJobs<R> jobs,
                                                             const R* __restrict__ U) {
  const int e = blockIdx.y;
  const SectorOperand& a = jobs.a[blockIdx.z];
  const SectorTables t = a.tab.at(e);
  const SectorPlan& p = *t.plan;
  const R* __restrict__ in = jobs.in[blockIdx.z] + e * a.in_bs;
  U += e * a.u_bs;
  R* __restrict__ out = elem_out<R, MODE>(jobs.out[blockIdx.z], e * a.out_bs);
  R* __restrict__ out_lo = elem_out<R, MODE>(jobs.lo[blockIdx.z], e * a.out_bs);
  unsigned* amax = a.amax ? a.amax + e * a.amax_bs : nullptr;
  const R uscale = (R)split_scale<MODE>(amax);
  extern __shared__ __align__(16) unsigned char fsm[];
  R* Us = (R*)fsm;      // [2][Db][NJ][Yp]: (charge of j, r, slot of j, slot of Y), zero past the last slots
  __shared__ OperandShared sh;
  const int Db = a.Db, lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
  const uint32_t mb = p.mb, nb = p.nb, na = p.na, mc = p.mc, mm = p.mm;
  const int parity = a.parity & p.odd;
  const int ny1 = odd_below(nb, a.cb), ny0 = a.cb - ny1, nj1 = odd_below(mb, Db), nj0 = Db - nj1;
  // slots of j: the counts that operand_run is built for (see the switch below)
  int NJp = max(nj0, nj1);
  if (NJM > 8) NJp = NJp <= 4 ? 4 : (NJp <= 8 ? NJp : (NJp <= 10 ? 10 : (NJp <= 12 ? 12 : 16)));
  const int Yp = (max(ny0, ny1) + 3) / 4 * 4;
  const int n0 = p.n3[0], n1 = p.n3[1];
  if (threadIdx.x < 2 * kMaxLeg) sh.jlist[threadIdx.x / kMaxLeg][threadIdx.x % kMaxLeg] = 0;   // unused slots: any valid j
  __syncthreads();
  if (threadIdx.x < kMaxLeg) {
    const int i = threadIdx.x;
    if (i < a.cb) sh.ylist[bit(nb, i)][bit(nb, i) ? odd_below(nb, i) : i - odd_below(nb, i)] = i;
    if (i < Db) sh.jlist[bit(mb, i)][bit(mb, i) ? odd_below(mb, i) : i - odd_below(mb, i)] = i;
  }
  for (int i = threadIdx.x; i < Db * Db * 2; i += blockDim.x) {
    const int g = i & 1, b1 = (i >> 1) % Db, b2 = (i >> 1) / Db;
    const int o1 = odd_below(mb, b1), o2 = odd_below(mb, b2);
    const int q1 = g ^ bit(mb, b1), Q = q1 ^ bit(mb, b2);       // charge of (b1', rest), of the summed index
    const int m0 = nj0 * n0 + nj1 * n1, m1 = nj0 * n1 + nj1 * n0;   // all runs of one b2 by the charge of (b1', rest)
    sh.base[b2][b1][g] = (b2 - o2) * (Q ? m1 : m0) + o2 * (Q ? m0 : m1) + (b1 - o1) * (q1 ? n1 : n0) + o1 * (q1 ? n0 : n1);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * Db * NJp * Yp; i += blockDim.x) {
    const int sl = i % Yp, js = (i / Yp) % NJp, r = (i / (Yp * NJp)) % Db, jc = i / (Yp * NJp * Db);
    const int y = jc ^ bit(mb, r);
    const bool in_u = sl < (y ? ny1 : ny0) && js < (jc ? nj1 : nj0);
    Us[i] = in_u ? U[sh.jlist[jc][js] * a.u_j + r * a.u_r + sh.ylist[y][sl]] * uscale : (R)0;
  }
  const int rows0 = p.row[0][a.x0 + a.xs] - p.row[0][a.x0];   // charge-0 rows of the slice
  const int roff0 = -p.row[0][a.x0], roff1 = rows0 - p.row[1][a.x0];
  const int c0n = (n0 + 63) / 64, per_seg = c0n + (n1 + 63) / 64;
  const uint32_t* rest = a.sideB ? t.kB : t.kA;
  const int K0 = p.K[0], K1 = p.K[1];
  unsigned long long tmax = 0;
  int buf = 0;
  for (int o = blockIdx.x; o < a.nouter; o += gridDim.x, buf ^= 1) {
    int r4 = o;
    const int m = r4 % a.Dm;
    r4 /= a.Dm;
    const int c1 = r4 % a.Dc;
    r4 /= a.Dc;
    const int c0 = r4 % a.Dc;
    const int X = r4 / a.Dc;
    const int qo = bit(na, a.x0 + X) ^ bit(mc, c0) ^ bit(mc, c1) ^ bit(mm, m) ^ parity;
    if (threadIdx.x < a.cb) {
      const int Y = threadIdx.x, q = bit(nb, Y);
      const uint32_t rk = t.row[((((int64_t)(a.x0 + X) * a.cb + Y) * a.Dc + c0) * a.Dc + c1) * a.Dm + m];
      sh.yrow[buf][q][q ? odd_below(nb, Y) : Y - odd_below(nb, Y)] =
          ((int64_t)(int)(rk & 0x7fffffffu) + (rk >> 31 ? roff1 : roff0)) * a.kps;
    }
    __syncthreads();
    if (MODE != kTTMMaxAbs && MODE != kTTMStore) {
      // zeros up to a whole k-block behind every row (a row of charge q holds the k of charge q + parity)
      for (int i = 2 * threadIdx.x; i < a.cb * a.kalign; i += 2 * blockDim.x) {
        const int Y = i / a.kalign, q = bit(nb, Y), KQ = (q ^ qo) ? K1 : K0;
        const int k = KQ + i % a.kalign;
        if (k >= (KQ + a.kalign - 1) / a.kalign * a.kalign) continue;
        const int sl = q ? odd_below(nb, Y) : Y - odd_below(nb, Y);
        sector_store2<MODE>(out, out_lo, sh.yrow[buf][q][sl] + k + (int64_t)(a.P > 1 ? k / (int)a.kps : 0) * (a.rows - 1) * a.kps,
                            (R)0, (R)0);
      }
    }
    const R* src = in + X * a.in_x + c0 * a.in_c0 + c1 * a.in_c1 + m * a.in_m;
    for (int it = warp; it < Db * per_seg; it += nwarp) {
      const int sg = it / per_seg, w = it - sg * per_seg;
      const int g = w >= c0n, i = (w - (g ? c0n : 0)) * 64 + 2 * lane;
      const bool live = i < (g ? n1 : n0);
      const uint2 ro = live ? *(const uint2*)(rest + (g ? n0 : 0) + i) : make_uint2(~0u, ~0u);
      const bool ok0 = ro.x != ~0u, ok1 = ro.y != ~0u;
      const R* xs = src + (int64_t)sg * a.in_seg;
      const R* x0 = xs + (ok0 ? ro.x : 0u);
      const R* x1 = xs + (ok1 ? ro.y : 0u);
      const int jc = qo ^ g ^ bit(mb, sg);                     // charge of the j with nonzero entries
      const int njc = jc ? nj1 : nj0;
#define HOTRG_RUN(N)                                                                                                 \
  operand_run<R, MODE, N>(x0, x1, ok0, ok1, live, i, jc, sg, g, mb, ny0, ny1, NJp, Yp, buf, Us, sh, a, out, out_lo, tmax)
      if constexpr (NJM <= 8) {
        switch (njc) {
          case 0: HOTRG_RUN(0); break;
          case 1: HOTRG_RUN(1); break;
          case 2: HOTRG_RUN(2); break;
          case 3: HOTRG_RUN(3); break;
          case 4: HOTRG_RUN(4); break;
          case 5: if constexpr (NJM >= 5) HOTRG_RUN(5); break;
          case 6: if constexpr (NJM >= 6) HOTRG_RUN(6); break;
          case 7: if constexpr (NJM >= 7) HOTRG_RUN(7); break;
          default: if constexpr (NJM >= 8) HOTRG_RUN(8); break;
        }
      } else {
        switch (njc) {
          case 0: case 1: case 2: case 3: case 4: HOTRG_RUN(4); break;   // unused slots: U is zero there
          case 5: HOTRG_RUN(5); break;
          case 6: HOTRG_RUN(6); break;
          case 7: HOTRG_RUN(7); break;
          case 8: HOTRG_RUN(8); break;
          case 9: case 10: HOTRG_RUN(10); break;
          case 11: case 12: HOTRG_RUN(12); break;
          default: HOTRG_RUN(16); break;
        }
      }
#undef HOTRG_RUN
    }
  }
  if (MODE == kTTMMaxAbs) {   // every thread gets here
    if constexpr (sizeof(R) == 8) merge_max(amax, __longlong_as_double((long long)tmax), a.amax_mul);
    else merge_max(amax, (double)__uint_as_float((unsigned)tmax), a.amax_mul);
  }
}

template <typename R>
cudaError_t launch_sector_operand(const SectorJobs<R>& jobs, const R* U, int ne, int mode, cudaStream_t st) {
  if (jobs.n < 1 || jobs.n > kMaxPassJobs) return cudaErrorInvalidValue;
  const SectorOperand& a = jobs.a[0];           // every job of a step has the same D_b and chi_b
  const size_t smem = (size_t)2 * a.Db * a.Db * ((a.cb + 3) / 4 * 4 + 4) * sizeof(R);   // a bound for any charges
  if (smem > (size_t)kSectorSmem) return cudaErrorInvalidValue;
  int64_t bx = 1;
  for (int i = 0; i < jobs.n; ++i) bx = jobs.a[i].nouter > bx ? jobs.a[i].nouter : bx;
  const int64_t share = 152 * 16 / ((int64_t)ne * jobs.n), cap = share > 32 ? share : 32;
  if (bx > cap) bx = cap;
  const dim3 g((unsigned)bx, ne, jobs.n);
  auto go = [&](auto kernel) -> cudaError_t {
    kernel<<<g, 256, smem, st>>>(jobs, U);
    return cudaGetLastError();
  };
  // the contracted leg's indices of one charge are at most D_b (all of one charge)
  auto pick = [&](auto mode_const) -> cudaError_t {
    constexpr int MODE = decltype(mode_const)::value;
    if (a.Db <= 4) return go(sector_operand_kernel<R, MODE, 4>);
    if (a.Db <= 8) return go(sector_operand_kernel<R, MODE, 8>);
    return go(sector_operand_kernel<R, MODE, 16>);
  };
  switch (mode) {
    case kTTMStore: return pick(std::integral_constant<int, kTTMStore>{});
    case kTTMMaxAbs: return pick(std::integral_constant<int, kTTMMaxAbs>{});
    case kTTMSplitF16: if constexpr (sizeof(R) == 4) return pick(std::integral_constant<int, kTTMSplitF16>{}); break;
    case kTTMSplitTF32: if constexpr (sizeof(R) == 4) return pick(std::integral_constant<int, kTTMSplitTF32>{}); break;
    case kTTMSplitOz: if constexpr (sizeof(R) == 8) return pick(std::integral_constant<int, kTTMSplitOz>{}); break;
  }
  return cudaErrorInvalidValue;
}
template cudaError_t launch_sector_operand<float>(const SectorJobs<float>&, const float*, int, int, cudaStream_t);
template cudaError_t launch_sector_operand<double>(const SectorJobs<double>&, const double*, int, int, cudaStream_t);

// ---------------------------------------------------------------------------- closing passes
// First closing pass: O3[Z][m][n] = sum_{c1, c2} U[c1, c2, Z] C[row(X, Y, c1, c1', mu1)][col(X', Y', c2, c2', mu2')]
// with m, n the ranked row groups (X, Y, c1', mu1) and (X', Y', c2', mu2'). A block takes NT column
// groups of one charge t and row groups of one charge r, four at a time: only the pairs (c1, c2) with
// q(c1) + q(c2) = s (s = r + t + the output's parity) and the Z of charge s are nonzero, the same for
// the whole block, so no lane is idle; the entries of the other Z are neither written nor read.
template <typename R, int NZ, int NT>
__global__ void __launch_bounds__(NT, NT == 128 ? (sizeof(R) * NZ > 64 ? 2 : 4) : 1)
    sector_close1_kernel(const R* __restrict__ C, const R* __restrict__ U, R* __restrict__ O3,
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
  const int ch0 = (n0 + NT - 1) / NT;
  const int tq = (int)blockIdx.x < ch0 ? 0 : 1;                 // charge of the column groups
  const int i0 = (tq ? (int)blockIdx.x - ch0 : (int)blockIdx.x) * NT;
  const int ncol = tq ? n1 : n0;
  if (i0 >= ncol) return;
  extern __shared__ __align__(16) unsigned char fsm[];
  R* Us = (R*)fsm;                                   // [2][Dc][Dc][NZ]: (charge of Z, c1, c2, slot), zero past the last slot
  int* rks = (int*)(Us + (size_t)2 * Dc * Dc * NZ);  // [Dc][NT] column of c2
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
  for (int i = tid; i < 2 * Dc * Dc * NZ; i += NT) {
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
      rks[c2 * NT + tid] = (int)(r & 0x7fffffffu) - p.row[r >> 31][a.x20];
    }
  }
  __syncthreads();
  const int rows0 = p.row[0][a.x0 + a.xs] - p.row[0][a.x0];
  const int mg0 = p.grp[0][a.x0 + a.xs] - p.grp[0][a.x0];   // charge-0 row groups of the slice
  const int64_t GR = (int64_t)a.xs * a.cb * inner, GC = (int64_t)a.xs2 * a.cb * inner;
  const int64_t ocol = (tq ? n0 : 0) + gi;
  const int parity = a.parity & p.odd;
  for (int rq = 0; rq < 2; ++rq) {
    const int gbase = p.grp[rq][a.x0], nrow = p.grp[rq][a.x0 + a.xs] - gbase;
    const int s = rq ^ tq ^ parity;
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
            const int col = rks[clist[jc][k + q] * NT + tid];
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
          const int col = rks[clist[jc][k] * NT + tid];
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
  const uint32_t mc = p.mc, nc = p.nc;
  const int parity = a.parity & p.odd;
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
    const int s = qm ^ qn ^ bit(nc, Z) ^ parity;
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
  const int64_t cols = (int64_t)a.xs2 * a.cb * a.Dc * a.Dm, rowg = (int64_t)a.xs * a.cb * a.Dc * a.Dm;
  // 128 threads fill small products and FP64 ones better (D_cut = 4: 20 -> 16 us, D = 6 FP64: 450 -> 330 us), 256
  // are faster on large FP32 ones (D_cut = 8: 993 us against 1085)
  const int NT = sizeof(R) == 4 && NZ > 4 && cols > 2048 ? 256 : 128;
  const size_t s1 = (size_t)2 * a.Dc * a.Dc * NZ * sizeof(R) + (size_t)a.Dc * NT * sizeof(int);
  const size_t s2 = (size_t)a.Dc * a.Dc * NZ * sizeof(R);
  if (s1 > (size_t)kSectorSmem) return cudaErrorInvalidValue;
  const int64_t bx = (cols + NT - 1) / NT + 1;
  int64_t by = (152 * 12 + bx * ne - 1) / (bx * ne);
  by = by < 1 ? 1 : by;
  by = by > (rowg + 7) / 8 ? (rowg + 7) / 8 : by;      // four row groups of one charge per step
  const dim3 g1((unsigned)bx, (unsigned)by, ne);
  int64_t b2 = (a.nfib + 255) / 256;
  const int64_t cap = 152 * 16 / ne > 8 ? 152 * 16 / ne : 8;
  if (b2 > cap) b2 = cap;
  const dim3 g2((unsigned)b2, ne);
  auto go = [&](auto k1, auto k2) -> cudaError_t {
    k1<<<g1, NT, s1, st>>>(C, U, O3, a);
    cudaError_t er = cudaGetLastError();
    if (er != cudaSuccess) return er;
    k2<<<g2, 256, s2, st>>>(O3, U, T, a);
    return cudaGetLastError();
  };
  if (NZ == 4) return go(sector_close1_kernel<R, 4, 128>, sector_close2_kernel<R, 4>);
  if (NT == 256) {
    if constexpr (sizeof(R) == 4) {
      if (NZ == 8) return go(sector_close1_kernel<R, 8, 256>, sector_close2_kernel<R, 8>);
      return go(sector_close1_kernel<R, 16, 256>, sector_close2_kernel<R, 16>);
    }
  }
  if (NZ == 8) return go(sector_close1_kernel<R, 8, 128>, sector_close2_kernel<R, 8>);
  return go(sector_close1_kernel<R, 16, 128>, sector_close2_kernel<R, 16>);
}
template cudaError_t launch_sector_close<float>(const float*, const float*, float*, float*, const SectorClose&, int,
                                                cudaStream_t);
template cudaError_t launch_sector_close<double>(const double*, const double*, double*, double*, const SectorClose&, int,
                                                 cudaStream_t);

// Once per device; a thread that finds another one at it waits until the attributes are set.
void sectors_prepare() {
  static std::once_flag once[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return;
  std::call_once(once[dev], [] {
    auto set = [](auto k) { cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSectorSmem); };
    set(sector_operand_kernel<double, kTTMStore, 16>);
    set(sector_operand_kernel<double, kTTMMaxAbs, 16>);
    set(sector_operand_kernel<double, kTTMSplitOz, 16>);
    set(sector_close1_kernel<float, 16, 128>);
    set(sector_close1_kernel<float, 16, 256>);
    set(sector_close1_kernel<double, 8, 128>);
    set(sector_close1_kernel<double, 16, 128>);
    set(sector_close2_kernel<double, 16>);
    cudaGetLastError();
  });
}

}  // namespace hotrg
