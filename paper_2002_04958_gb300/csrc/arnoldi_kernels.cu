// arnoldi_kernels.cu -- one FGMRES orthogonalisation (modified Gram-Schmidt of
// w against the basis, then the normalisation) as one launch: a cooperative
// grid, or one cluster where there are few unknowns.
//
// Modified Gram-Schmidt takes h_i = <v_i, w - sum_{k<i} h_k v_k>, one grid-wide
// reduction after the other.  With l_ik = <v_i, v_k> the same coefficients
// solve the unit lower triangular system
//     h_i + sum_{k<i} l_ik h_k = <v_i, w>
// (the compact-WY form of modified Gram-Schmidt; Swirydowicz, Langou, Ananthan,
// Yang, Thomas, "Low synchronization Gram-Schmidt and generalized minimal
// residual algorithms", Numer. Linear Algebra Appl. 2021), so one pass over the
// basis gives every <v_i, w>, and with it the new row l_j. of the Gram matrix,
// and a second pass subtracts sum_i h_i v_i: two grid barriers and 16 bytes per
// entry of the basis, where a pass per basis vector takes one barrier (or
// launch) and 32 bytes each.
//
// A dot product on the FP64 pipe costs a warp 20 SM clocks per multiply-add
// here (15.7 G warp instructions/s over 152 SMs), more than the 12 clocks that
// the 256 bytes it reads take from HBM, and the first pass has two of them per
// entry.  So that pass multiplies on the integer pipe, exactly: the entries of
// a unit (32 lanes x K) are aligned to the unit's largest exponent and split
// into two signed limbs (29 + 29 bits below the largest, a half-unit midpoint
// for what is cut off), the four limb products are summed in 64-bit integers,
// folded across the warp as integers, and only the unit's sums become FP64.
// The rounding against binary64 products is below theirs: 2^-57 of the unit's
// largest entry per element, of either sign.
//
// Measured per call with 16 vectors, against the streaming kernels: 3,072
// unknowns 17.6 / 110.9 us, 148,074 33 / 178 us, 3.1 M 227 / 394 us, 19.5 M
// 1160 / 1617 us; there the first pass takes 23 us a vector (its 156 MB at the
// copy bandwidth) and the second 39 us, its FP64 issue slots.  The second pass
// on the integer pipe was no faster (34 us a vector, and more per call).
#include "mgd_internal.cuh"

#include <cooperative_groups.h>

namespace mgd {

namespace cg = cooperative_groups;

constexpr int kGsWarps = 12;
constexpr int kGsThreads = 32 * kGsWarps;
constexpr int kGsMinWarps = 8;  // busy warps to a block before there is another block

__device__ __forceinline__ int exp_of(int hi) { return (hi >> 20) & 0x7ff; }

// |x| = (53-bit m) 2^(e - 1075) as (h 2^29 + l) 2^(eref - 1082), eref >= e + 2,
// both limbs with x's sign; l is odd: the midpoint of the cut-off part
__device__ __forceinline__ void split_limbs(double x, int eref, int& h, int& l) {
  const int hi = __double2hiint(x);
  const unsigned r = min((unsigned)(eref - exp_of(hi)), 63u);
  unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(x);
  m = (m << 7) >> r;
  const int sg = (hi >> 31) | 1;
  h = (int)(m >> 29) * sg;
  l = (int)(((unsigned)m & 0x1fffffffu) | 1u) * sg;
}

// the three sums of a limb dot product, folded over the warp into four 27-bit
// limbs (the last one signed) of  hh 2^29 + x + ll 2^-29
struct LimbSum {
  long long hh = 0, x = 0, ll = 0;
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {
    hh += (long long)ah * bh;
    x += (long long)ah * bl;
    x += (long long)al * bh;
    ll += (long long)al * bl;
  }
  __device__ __forceinline__ int4 fold() const {
    const __int128 t = ((__int128)hh << 29) + x + (ll >> 29);
    constexpr unsigned M = (1u << 27) - 1;
    int4 f;
    f.x = (int)__reduce_add_sync(0xffffffffu, (unsigned)t & M);
    f.y = (int)__reduce_add_sync(0xffffffffu, (unsigned)(t >> 27) & M);
    f.z = (int)__reduce_add_sync(0xffffffffu, (unsigned)(t >> 54) & M);
    f.w = __reduce_add_sync(0xffffffffu, (int)(t >> 81));
    return f;
  }
};

__device__ __forceinline__ double unfold(const int4& f) {
  const long long lo = ((long long)(unsigned)f.y << 27) + (unsigned)f.x;
  const long long hi = ((long long)f.w << 27) + (unsigned)f.z;
  return fma((double)hi, 0x1p54, (double)lo);
}

// V: nv basis vectors (leading dimension ldv), each unit's largest biased
// exponent in vexp[i * nunits + u]; gram: l_ik at gram[k * 32 + i], rows < nv-1
// given, row nv-1 written by block 0.  Writes h[0..nv-1], *nrm2 = ||w'||^2 and
// vout = w' / ||w'|| with its exponents; w is only read.
template <int K, bool CLUSTER>
__global__ void __launch_bounds__(kGsThreads, 1)
    k_gram_schmidt(int n, const double* __restrict__ V, long long ldv, int nv, const double* __restrict__ w,
                   int* vexp, int nunits, int share_of_short, double* gram, double* __restrict__ h,
                   double* __restrict__ nrm2, double* part, double* vout) {
  __shared__ int4 s_fold[kGsWarps][32][2];
  __shared__ double s_gram[32 * 32];
  __shared__ double s_sum[kGsWarps][64];
  __shared__ double s_dot[64], s_h[32], s_red[kGsWarps];
  auto sync = [] {
    if (CLUSTER) cg::this_cluster().sync();  // (one cluster: release and acquire of global memory within it)
    else cg::this_grid().sync();
  };
  // (the next launch only once the ones before this are over: three deep, a
  // kernel could start while the step's first ones still read)
  if (CLUSTER) MGD_PDL_ENTRY();
  constexpr int U = 32 * K, H = K / 2, UI = K >= 16 ? 2 : K >= 8 ? 4 : 8;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  // warps are numbered across the blocks, so that units spread over all SMs
  const int nb = gridDim.x, gw = warp * nb + blockIdx.x, nw = nb * kGsWarps;
  const int j = nv - 1;
  for (int q = t; q < 32 * 32; q += kGsThreads) s_gram[q] = gram[q];

  // <v_i, w> and <v_i, v_j>, lane i holding those of v_i; `share` warps take a
  // unit, each every share-th vector
  double acc_w = 0.0, acc_g = 0.0;
  const int share = K <= 4 ? share_of_short : 1;
  const int i0 = gw % share;
  for (int u = gw / share; u < nunits; u += nw / share) {
    const long long e0 = (long long)u * U + lane;
    const int ei = lane < nv ? vexp[(size_t)lane * nunits + u] : 0;
    int ah[K], al[K], bh[K], bl[K];
    int ew = 0;
    const int ej = __shfl_sync(0xffffffffu, ei, j);
    {
      double x[K], y[K];
#pragma unroll
      for (int q = 0; q < K; ++q) {
        const bool ok = e0 + 32 * q < n;
        x[q] = ok ? __ldcs(w + e0 + 32 * q) : 0.0;
        y[q] = ok ? V[(long long)j * ldv + e0 + 32 * q] : 0.0;
      }
#pragma unroll
      for (int q = 0; q < K; ++q) ew = max(ew, exp_of(__double2hiint(x[q])));
      ew = __reduce_max_sync(0xffffffffu, ew);
#pragma unroll
      for (int q = 0; q < K; ++q) {
        split_limbs(x[q], ew + 2, ah[q], al[q]);
        if (exp_of(__double2hiint(x[q])) == 0) ah[q] = al[q] = 0;
        split_limbs(y[q], ej + 2, bh[q], bl[q]);
        if (exp_of(__double2hiint(y[q])) == 0) bh[q] = bl[q] = 0;
      }
    }
    // (past n these read the next vector or the padding after the basis, times zero limbs of w and v_j)
    const double* v = V + e0;
    double va[H], vb[H];
    auto load = [&](double (&d)[H], int i, int q0) {
#pragma unroll
      for (int q = 0; q < H; ++q) d[q] = v[(long long)i * ldv + 32 * (q0 + q)];
    };
    auto take = [&](const double (&d)[H], int i, int q0, LimbSum& dw, LimbSum& dg) {
      const int e = __shfl_sync(0xffffffffu, ei, i) + 3;
#pragma unroll
      for (int q = 0; q < H; ++q) {
        int vh, vl;
        split_limbs(d[q], e, vh, vl);
        dw.add(vh, vl, ah[q0 + q], al[q0 + q]);
        dg.add(vh, vl, bh[q0 + q], bl[q0 + q]);
      }
    };
    if (i0 < nv) {
      load(va, i0, 0);
      load(vb, i0, H);
    }
#pragma unroll 1
    for (int i = i0; i < nv; i += share) {
      LimbSum dw, dg;
      take(va, i, 0, dw, dg);
      if (i + share < nv) load(va, i + share, 0);
      take(vb, i, H, dw, dg);
      if (i + share < nv) load(vb, i + share, H);
      const int4 fw = dw.fold(), fg = dg.fold();
      if (lane == 0) {
        s_fold[warp][i][0] = fw;
        s_fold[warp][i][1] = fg;
      }
    }
    __syncwarp();
    if (lane < nv && lane % share == i0 && ei >= 70) {  // a unit of v_i below 2^-953 adds nothing
      // one unit of the folded sums is 2^(exponents - 2 * 1023 - 84)
      const double s = 0x1p-84 * __hiloint2double(ei << 20, 0);
      acc_w += unfold(s_fold[warp][lane][0]) * s * __hiloint2double(ew << 20, 0);
      acc_g += unfold(s_fold[warp][lane][1]) * s * __hiloint2double(ej << 20, 0);
    }
    __syncwarp();
  }
  s_sum[warp][lane] = acc_w;
  s_sum[warp][32 + lane] = acc_g;
  __syncthreads();
  if (t < 64 && (t & 31) < nv) {
    double s = 0.0;
    for (int q = 0; q < kGsWarps; ++q) s += s_sum[q][t];
    part[(size_t)t * nb + blockIdx.x] = s;
  }
  sync();

  // every block: the dot products from the per-block sums (the same order in
  // all), then the triangular system, a row per lane
  for (int p = warp; p < 2 * nv; p += kGsWarps) {
    const int row = p < nv ? p : 32 + p - nv;
    double s = 0.0;
    for (int b = lane; b < nb; b += 32) s += __ldcg(part + (size_t)row * nb + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) s_dot[row] = s;
  }
  __syncthreads();
  if (warp == 0) {
    if (lane < j) s_gram[lane * 32 + j] = s_dot[32 + lane];
    __syncwarp();
    double hv = lane < nv ? s_dot[lane] : 0.0;
    for (int k = 0; k < j; ++k) {
      const double hk = __shfl_sync(0xffffffffu, hv, k);
      if (lane > k && lane < nv) hv -= s_gram[k * 32 + lane] * hk;
    }
    s_h[lane] = hv;
    if (blockIdx.x == 0) {
      if (lane < nv) h[lane] = hv;
      if (lane < j) gram[lane * 32 + j] = s_gram[lane * 32 + j];
    }
  }
  __syncthreads();

  // w' = w - sum_i h_i v_i and ||w'||^2
  double ss = 0.0;
  for (int u = gw; u < nunits; u += nw) {
    const long long e0 = (long long)u * U + lane;
    double x[K];
#pragma unroll
    for (int q = 0; q < K; ++q) x[q] = e0 + 32 * q < n ? __ldcs(w + e0 + 32 * q) : 0.0;
#pragma unroll UI
    for (int i = 0; i < nv; ++i) {
      const double hi = s_h[i];
      const double* v = V + (long long)i * ldv + e0;
#pragma unroll
      for (int q = 0; q < K; ++q)
        if (e0 + 32 * q < n) x[q] -= hi * __ldcs(v + 32 * q);
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
      ss += x[q] * x[q];
      if (e0 + 32 * q < n) vout[e0 + 32 * q] = x[q];
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if (lane == 0) s_red[warp] = ss;
  __syncthreads();
  if (t == 0) {
    double s = 0.0;
    for (int q = 0; q < kGsWarps; ++q) s += s_red[q];
    part[(size_t)64 * nb + blockIdx.x] = s;
  }
  sync();
  double nn = 0.0;  // every warp for itself, in the same order
  for (int b = lane; b < nb; b += 32) nn += __ldcg(part + (size_t)64 * nb + b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) nn += __shfl_xor_sync(0xffffffffu, nn, o);
  if (blockIdx.x == 0 && t == 0) *nrm2 = nn;
  const double hn = sqrt(nn), inv = hn != 0.0 ? 1.0 / hn : 0.0;
  // the normalisation, from the units written last (still in L2) to the first
  const int mine = gw < nunits ? (nunits - 1 - gw) / nw : -1;
  for (int k = mine; k >= 0; --k) {
    const int u = gw + k * nw;
    const long long e0 = (long long)u * U + lane;
    double x[K];
    int e = 0;
#pragma unroll
    for (int q = 0; q < K; ++q) x[q] = e0 + 32 * q < n ? vout[e0 + 32 * q] * inv : 0.0;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      e = max(e, exp_of(__double2hiint(x[q])));
      if (e0 + 32 * q < n) vout[e0 + 32 * q] = x[q];
    }
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) vexp[(size_t)nv * nunits + u] = e;
  }
}

// the unit exponents of one vector (a cycle's first basis vector)
__global__ void __launch_bounds__(kThreads) k_unit_exponents(int n, int unit, const double* __restrict__ v, int* vexp,
                                                             int nunits) {
  MGD_PDL_ENTRY();
  const int u = (blockIdx.x * kThreads + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (u >= nunits) return;
  const long long e1 = min((long long)n, (long long)(u + 1) * unit);
  int e = 0;
  for (long long i = (long long)u * unit + lane; i < e1; i += 32) e = max(e, exp_of(__double2hiint(v[i])));
  e = __reduce_max_sync(0xffffffffu, e);
  if (lane == 0) vexp[u] = e;
}

static const void* gs_kernel(int K) {
  return K == 2 ? (const void*)k_gram_schmidt<2, false> : K == 4 ? (const void*)k_gram_schmidt<4, false>
       : K == 8 ? (const void*)k_gram_schmidt<8, false> : (const void*)k_gram_schmidt<16, false>;
}

// Few unknowns: what a step takes is the launch and the two barriers, so its
// blocks are one cluster.  Its hardware barrier takes 0.3-0.5 us where the
// grid's takes some 2, and unlike a cooperative grid it may start on the
// product's heels (programmatic dependent launch).  A step on 3,072 unknowns
// 39.0 -> 35.4 us.  Sixteen SMs' FP64 pipes set the line: the kernel alone with
// 1 / 8 / 16 / 30 vectors, grid against cluster: 3,072 unknowns 14.5 / 16.6 /
// 20.5 / 24.8 against 12.5 / 14.6 / 17.6 / 24.8 us; 8,192 unknowns 14.5 / 18.5 /
// 20.7 / 28.5 against 12.4 / 16.6 / 20.7 / 30.9; 24,576 unknowns 16.8 / 20.7 /
// 24.8 / 32.8 against 16.4 / 24.8 / 35.7 / 55.5.
constexpr int kGsClusterMax = 8192;

static cudaLaunchConfig_t gs_cluster_config(int blocks, cudaLaunchAttribute (&attr)[2], cudaStream_t s) {
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = blocks;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kGsThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = tl_pdl ? 2 : 1;
  return cfg;
}

// the largest cluster of the kernel that the device takes: 16 blocks (a size
// that has to be allowed first), else the portable 8, else 0
static int gs_cluster_blocks() {
  for (int cs : {16, 8}) {
    int fits = 0;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = gs_cluster_config(cs, attr, nullptr);
    cfg.numAttrs = 1;
    if ((cs <= 8 ||
         cudaFuncSetAttribute(k_gram_schmidt<2, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
             cudaSuccess) &&
        cudaOccupancyMaxActiveClusters(&fits, k_gram_schmidt<2, true>, &cfg) == cudaSuccess && fits > 0)
      return cs;
    cudaGetLastError();
  }
  return 0;
}

GsPlan gs_plan(int n) {
  GsPlan p;
  int dev = 0, sms = 0, coop = 0, per = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)) {
    cudaGetLastError();
    return p;
  }
  if (!coop || sms <= 0 || n <= 0) return p;
  const long long lanes = (long long)sms * kGsThreads;
  if (n <= kGsClusterMax) {
    p.K = 2;
    const int most = gs_cluster_blocks();
    if (most > 0) {
      p.nunits = cdiv(n, 32 * p.K);
      while (p.share < 8 && p.nunits * p.share * 2 <= most * kGsWarps) p.share *= 2;
      p.nb = 1;
      while (p.nb < most && p.nb * kGsMinWarps < p.nunits * p.share) p.nb *= 2;
      p.cluster = true;
      return p;
    }
  }
  // long units fold less often, short ones keep every warp busy: the shortest
  // that still gives each warp one unit, then 256 entries while 512 would leave
  // a warp five or fewer (1 M unknowns, 16 vectors: 100 us against 128 us;
  // 19.5 M: 1280 against 1160)
  const int K = n <= 2 * lanes ? 2 : n <= 4 * lanes ? 4 : n <= 80 * lanes ? 8 : 16;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, gs_kernel(K), kGsThreads, 0) != cudaSuccess || per < 1) {
    cudaGetLastError();
    return p;
  }
  p.K = K;
  p.nunits = cdiv(n, 32 * K);
  // a short vector leaves warps without a unit: several share one (3,072
  // unknowns, 30 vectors: 35 -> 25 us)
  p.share = 1;
  while (K <= 4 && p.share < 8 && (long long)p.nunits * p.share * 2 <= (long long)sms * kGsWarps) p.share *= 2;
  p.nb = std::min(sms, cdiv((long long)p.nunits * p.share, kGsMinWarps));
  return p;
}

void launch_unit_exponents(const GsPlan& p, int n, const double* v, int* vexp, cudaStream_t s) {
  launch_k(k_unit_exponents, dim3(cdiv(32LL * p.nunits, kThreads)), dim3(kThreads), 0, s, n, 32 * p.K, v, vexp,
           p.nunits);
  MGD_LAUNCH_CHECK();
}

void launch_gram_schmidt(const GsPlan& p, int n, const double* V, long long ldv, int nv, const double* w, int* vexp,
                         double* gram, double* h, double* nrm2, double* part, double* vout, cudaStream_t s) {
  int nunits = p.nunits, share = p.share;
  if (p.cluster) {
    cudaLaunchAttribute attr[2];
    const cudaLaunchConfig_t cfg = gs_cluster_config(p.nb, attr, s);
    MGD_CUDA(cudaLaunchKernelEx(&cfg, k_gram_schmidt<2, true>, n, V, ldv, nv, w, vexp, nunits, share, gram, h, nrm2,
                                part, vout));
    MGD_LAUNCH_CHECK();
    return;
  }
  void* args[] = {(void*)&n, (void*)&V, (void*)&ldv, (void*)&nv, (void*)&w, (void*)&vexp, (void*)&nunits,
                  (void*)&share, (void*)&gram, (void*)&h, (void*)&nrm2, (void*)&part, (void*)&vout};
  MGD_CUDA(cudaLaunchCooperativeKernel(gs_kernel(p.K), dim3(p.nb), dim3(kGsThreads), args, 0, s));
  MGD_LAUNCH_CHECK();
}

}  // namespace mgd
