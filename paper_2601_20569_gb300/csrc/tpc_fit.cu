// Track merging and the final fit (Sec. 2 "track merging and track fit",
// Sec. 3 Phases I and II):
//   a7  sector refit of every accepted tracklet and mutual-best merging of
//       track ends inside a sector and between adjacent sectors of one half;
//   a8  space-charge correction of clusters with a cubic B-spline map;
//   a9  three-iteration linearised Kalman fit: iteration 1 inward stores the
//       predicted (y,z) and covariance per station, iteration 2 outward
//       interpolates and flags outliers, iteration 3 inward refits;
//   a10 Phase II re-attachment on the inner rows: candidates within the
//       interpolation cut, second ambiguity solving in cand_k rounds;
//   a11 output compaction and cluster-to-track attachment.
// Compiled twice (strict / fast) like the sector kernels.
#include <cuda_runtime.h>

#include <cstdint>

#include "tpc_kernels.h"
#include "tpc_model.cuh"
#include "tpc_util.cuh"

namespace tpc {
namespace TPC_NS {

namespace {

// --------------------------------------------------------- a8 distortion map
__device__ __forceinline__ void spline_w(float f, float* w) {
  const float g = 1.0f - f;
  const float f2 = f * f, f3 = f2 * f;
  w[0] = g * g * g / 6.0f;
  w[1] = (3.0f * f3 - 6.0f * f2 + 4.0f) / 6.0f;
  w[2] = (-3.0f * f3 + 3.0f * f2 + 3.0f * f + 1.0f) / 6.0f;
  w[3] = f3 / 6.0f;
}

__device__ __forceinline__ void spline_span(float t, int n, int& i, float& f) {
  const float tmax = (float)(n - 3);
  if (t < 0.0f) t = 0.0f;
  if (t > tmax) t = tmax;
  i = (int)floorf(t);
  if (i > n - 4) i = n - 4;
  f = t - (float)i;
}

struct SplinePt {
  int ip, ir, iz;
  float wp[4], wr[4], wz[4];
};

// x^2 + y^2 of a map point.  Strict mode rounds every operation; fast mode fuses
// one product into the sum.  The refit states which one (kXFirst), so that its
// values do not hang on the order in which the compiler meets the products.
template <bool kXFirst>
__device__ __forceinline__ float square_sum(float x, float y) {
#ifdef TPC_FAST_ARITH
  if (kXFirst) return __fmaf_rn(x, x, __fmul_rn(y, y));
#endif
  return x * x + y * y;
}

template <bool kXFirst = false>
__device__ __forceinline__ SplinePt spline_point(const MapDev& M, const KParams& P, int sector,
                                                 float x, float y, float zdrift) {
  SplinePt sp;
  const int sphi = sector % P.n_phi;
  const float u = ((float)sphi + 0.5f) + 0.5f * (y / x) / P.tan_half;
  const float tp = u * M.phi_scale - 0.5f;
  sp.ip = (int)floorf(tp);
  const float fp = tp - (float)sp.ip;
  const float r = sqrtf(square_sum<kXFirst>(x, y));
  float fr, fz;
  spline_span((r - M.rmin) * M.r_scale, M.nr, sp.ir, fr);
  float zc = zdrift;
  if (zc < M.zmin) zc = M.zmin;
  if (zc > M.zmax) zc = M.zmax;
  spline_span((zc - M.zmin) * M.z_scale, M.nz, sp.iz, fz);
  spline_w(fp, sp.wp);
  spline_w(fr, sp.wr);
  spline_w(fz, sp.wz);
  return sp;
}

__device__ __forceinline__ int phi_index(int ip, int e, int nphi) {
  return ((ip - 1 + e) % nphi + nphi) % nphi;
}

template <bool kXFirst = false>
__device__ __forceinline__ void map_eval(const MapDev& M, const KParams& P, int sector, float x,
                                         float y, float zdrift, float* D) {
  D[0] = D[1] = D[2] = 0.0f;
  if (!M.on) return;
  const SplinePt sp = spline_point<kXFirst>(M, P, sector, x, y, zdrift);
  int pidx[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) pidx[e] = phi_index(sp.ip, e, M.nphi);
  // one 16-byte load per control point gives its three components (the packed
  // map of 18 x 16 x 20 control points, 92 KB, stays in L1); each component's sum
  // runs in the order z, r, phi
  // (the z loop stays a loop, its weights handed down: 64 loads in flight at once
  // would hold 160 registers)
  float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f;
  float wz = sp.wz[0], wz1 = sp.wz[1], wz2 = sp.wz[2];
#pragma unroll 1
  for (int a = 0; a < 4; ++a) {
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const float wzr = wz * sp.wr[b];
      const float4* row = M.c4 + ((long)(sp.iz + a) * M.nr + (sp.ir + b)) * M.nphi;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 v = __ldg(row + pidx[e]);
        const float w = wzr * sp.wp[e];
        a0 = a0 + w * v.x;
        a1 = a1 + w * v.y;
        a2 = a2 + w * v.z;
      }
    }
    wz = wz1;
    wz1 = wz2;
    wz2 = sp.wz[3];
  }
  D[0] = a0;
  D[1] = a1;
  D[2] = a2;
}

// The map's control points with their components side by side, packed anew for
// every call (the caller may change the coefficients between calls).
__global__ void k_map_pack(MapDev M, float4* c4) {
  const long n = (long)M.nz * M.nr * M.nphi;
  for (long i = (long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long)gridDim.x * blockDim.x)
    c4[i] = make_float4(M.c[i], M.c[n + i], M.c[2 * n + i], 0.0f);
}

// Corrected measurement projected back onto the pad row along the reference.
__device__ __forceinline__ bool corrected(const MapDev& M, const KParams& P, int sector, float x,
                                          float y, float z, float z0, const float* ref, float& my,
                                          float& mz) {
  float D[3];
  map_eval(M, P, sector, x, y, z - z0, D);
  my = y + D[1];
  mz = z + D[2];
  if (D[0] != 0.0f) {
    StepJ st;
    if (!helix_step(ref, D[0], P, st, P.fit_max_snp)) return false;
    my = my - (st.p0 - ref[0]);
    mz = mz - (st.p1 - ref[1]);
  }
  return true;
}

// ------------------------------------------------------ a7 sector refit
__device__ __forceinline__ unsigned long long pack_chi_key(float chi2, int key) {
  return ((unsigned long long)f2o(chi2) << 32) | (unsigned long long)(unsigned)key;
}

// Compaction of accepted tracklets into the sector-track list (tracklet order).
__global__ void k_acc_count(FrameDev F) {
  __shared__ int sh[32];
  const int nst = min(F.cnt->n_starts, (int)F.cap_tl);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int f = (!F.cnt->err && i < nst && F.tl_acc[i]) ? 1 : 0;
  int tot;
  block_exscan(f, sh, &tot);
  if (threadIdx.x == 0) F.scan_tmp[blockIdx.x] = tot;
}

__global__ void k_acc_write(FrameDev F) {
  __shared__ int sh[32];
  const int nst = min(F.cnt->n_starts, (int)F.cap_tl);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int f = (!F.cnt->err && i < nst && F.tl_acc[i]) ? 1 : 0;
  int tot;
  const int ex = block_exscan(f, sh, &tot);
  // room for the track's kept-cluster positions: one atomic per warp (the
  // layout of the position array is arbitrary; every track reads its own range)
  const int nk = f ? F.tl_nkept[i] : 0;
  const int lane = threadIdx.x & 31;
  int incl = nk;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  int base = 0;
  if (lane == 31 && incl > 0) base = atomicAdd(&F.cnt->n_pos, incl);
  base = __shfl_sync(0xffffffffu, base, 31);
  const unsigned act = __ballot_sync(0xffffffffu, f != 0);
  if (f) {
    const int j = F.scan_tmp[blockIdx.x] + ex;
    F.st_tl[j] = i;
    F.st_off[j] = base + incl - nk;
    // scheduling bucket of the sector refit: most clusters first (the lanes
    // of one bucket take their places with one atomic; the order inside a
    // bucket only schedules the refit)
    const int b = kOrdBuckets - 1 - min(kOrdBuckets - 1, nk);
    const unsigned peers = __match_any_sync(act, b);
    const int leader = __ffs(peers) - 1;
    int slot = 0;
    if (lane == leader) slot = atomicAdd(&F.st_ord_cnt[b], __popc(peers));
    slot = __shfl_sync(peers, slot, leader);
    F.st_obucket[j] = b;
    F.st_oslot[j] = slot + __popc(peers & ((1u << lane) - 1u));
  }
}

// Positions (pad-row x, y, z) of every sector track's kept clusters, in
// kept order, gathered once so that the two passes of the sector refit read
// each track's clusters as one contiguous run.
__global__ void k_st_gather(FrameDev F, KParams P) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  if (F.cnt->n_pos > F.cap_pos) {
    if (blockIdx.x == 0 && threadIdx.x == 0) atomicOr(&F.cnt->err, kErrCapPos);
    return;
  }
  const int NR = P.n_rows;
  __shared__ float rx[kMaxRows];
  for (int r = threadIdx.x; r < NR; r += blockDim.x) rx[r] = F.row_x[r];
  __syncthreads();
  // One warp per 32 consecutive tracks (fewer where that would leave warps
  // without work): lane j loads track j's tracklet, length and output place
  // (all lanes at once), then the warp takes the tracks one by one, its lanes reading the whole kept list (up to kMaxRows
  // entries, all loads issued before the positions they address) and
  // writing the positions 32 at a time.
  constexpr int kChunks = (kMaxRows + 31) / 32;
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (blockDim.x >> 5);
  const int per = warp_share(ns, nw);
  for (int j0 = per * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); j0 < ns;
       j0 += per * nw) {
    int ti = 0, nk = 0, off = 0;
    if (lane < per && j0 + lane < ns) {
      ti = F.st_tl[j0 + lane];
      nk = F.tl_nkept[ti];
      off = F.st_off[j0 + lane];
    }
    for (int j = 0; j < per; ++j) {
      const int tj = __shfl_sync(0xffffffffu, ti, j);
      const int nj = __shfl_sync(0xffffffffu, nk, j);
      const int oj = __shfl_sync(0xffffffffu, off, j);
      const int* K = F.tl_kept + (long)tj * kMaxRows;
      float4* out = F.st_pos + oj;
      int c[kChunks];
#pragma unroll
      for (int u = 0; u < kChunks; ++u) {
        const int m = lane + 32 * u;
        c[u] = m < nj ? K[m] : -1;
      }
      float2 yz[kChunks];
      int rr[kChunks];
#pragma unroll
      for (int u = 0; u < kChunks; ++u) {
        yz[u] = c[u] >= 0 ? F.syz[c[u]] : make_float2(0.0f, 0.0f);
        rr[u] = c[u] >= 0 ? F.srow[c[u]] : 0;
      }
#pragma unroll
      for (int u = 0; u < kChunks; ++u)
        if (c[u] >= 0)
          out[lane + 32 * u] =
              make_float4(rx[rr[u] % NR], yz[u].x, yz[u].y, __int_as_float(rr[u]));
    }
  }
}

// Sector refit as a per-lane state machine: every loop iteration is one step
// (propagate to a kept cluster, update) of the lane's current track, and a
// lane whose track ends takes the next one from the work queue.  A track's
// 2 nk steps run outward over its kept clusters (innermost first), then, with
// reset covariance, inward over the same ones; the next position is requested
// one step ahead of the filter.  One loop body for both passes and all tracks,
// because what bounds the kernel is the serial chain of a track's steps: as
// two nested loops per track the lanes of a warp did not reconverge between
// tracks and passes of unequal length, and a step cost 5 us instead of 0.8.
__global__ void __launch_bounds__(256) k_sector_refit(FrameDev F, KParams P, int stat) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  const int NR = P.n_rows;
  bool busy = false, inward = false, first = true;
  int i = 0, sec = 0, nk = 0, left = 0;
  const float4* pos = nullptr;
  float4 nxt;
  Trk<float> t;
  for (;;) {
    if (!busy) {
      const int q = next_item(&F.cnt->queue[kQSectorRefit], first, stat);
      if (q >= ns) break;
      i = F.st_order[q];
      const int ti = F.st_tl[i];
      nk = F.tl_nkept[ti];
      pos = F.st_pos + F.st_off[i];  // kept clusters, outermost first
      const int rs0 = __float_as_int(pos->w);
      pos += nk - 1;
      nxt = *pos;
      const int rs = __float_as_int(nxt.w);
      sec = rs / NR;
      F.st_key[i] = F.sid[F.starts[ti]];
      F.st_sector[i] = sec;
      F.st_rmin[i] = rs % NR;
      F.st_rmax[i] = rs0 % NR;
      F.st_next[i] = -1;
      F.st_hasprev[i] = 0;
      F.st_bestB[i] = -1;
      F.st_bestA[i] = ~0ull;
      F.st_xbestB[i] = -1;
      F.st_xbestA[i] = ~0ull;
      F.st_dz[i] = 0.0f;
#pragma unroll
      for (int k = 0; k < 5; ++k) t.p[k] = F.tl_par[(long)ti * 5 + k];
      t.x = F.tl_x[ti];
      reset_cov(t.c, P);
      left = nk;
      inward = false;
      busy = true;
      continue;
    }
    const float4 cur = nxt;
    if (--left > 0) {  // (the inward pass starts at the cluster the outward one ends on)
      pos += inward ? 1 : -1;
      nxt = *pos;
    }
    if (!propagate(t, cur.x, P, P.fit_max_snp)) {
      F.st_ok[i] = 0;
      busy = false;
      continue;
    }
    update(t, residual(t, cur.y, cur.z, P));
    if (left > 0) continue;
    put_state((inward ? F.st_ie : F.st_oe) + (long)i * kStateF, t, sec);
    if (inward) {
      F.st_ok[i] = 1;
      busy = false;
    } else {
      reset_cov(t.c, P);
      left = nk;
      inward = true;
    }
  }
}

// z range of each sector (from the row statistics of the grid build).
constexpr float kMergeBinCm = 8.0f;

__global__ void k_sector_zrange(FrameDev F, KParams P) {
  const int s = blockIdx.x;
  __shared__ unsigned lo, hi;
  if (threadIdx.x == 0) { lo = 0xFFFFFFFFu; hi = 0u; }
  __syncthreads();
  for (int r = threadIdx.x; r < P.n_rows; r += blockDim.x) {
    const int rr = s * P.n_rows + r;
    if (F.row_cnt[rr] > 0) {
      atomicMin(&lo, F.row_zmin[rr]);
      atomicMax(&hi, F.row_zmax[rr]);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float zl = 0.0f, zh = 1.0f;
    if (hi >= lo && hi != 0u) { zl = o2f(lo); zh = o2f(hi); }
    F.sec_zlo[s] = zl;
    // (bins of at least kMergeBinCm: the search windows are 10-30 cm long)
    F.sec_zinv[s] = zh > zl ? fminf((float)kMergeZ / (zh - zl), 1.0f / kMergeBinCm) : 0.0f;
  }
}

// Merge candidate index: inner ends binned by (sector, z, innermost row), so
// that the rows a pair test accepts form one contiguous range per z bin.
__device__ __forceinline__ int merge_zbin(const FrameDev& F, int s, float z) {
  return clampi((int)floorf((z - F.sec_zlo[s]) * F.sec_zinv[s]), 0, kMergeZ - 1);
}
__device__ __forceinline__ int merge_bin(const FrameDev& F, int nrows, int s, int r, float z) {
  return (s * kMergeZ + merge_zbin(F, s, z)) * nrows + r;
}

__global__ void k_ie_hist(FrameDev F, KParams P) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ns; i += gridDim.x * blockDim.x) {
    // (an inner end linked by the edge following takes no part in the merging)
    if (!F.st_ok[i] || F.st_hasprev[i]) { F.ie_bin[i] = -1; continue; }
    const int b = merge_bin(F, P.n_rows, F.st_sector[i], F.st_rmin[i],
                            F.st_ie[(long)i * kStateF + 1]);
    F.ie_bin[i] = b;
    F.ie_slot[i] = atomicAdd(&F.ie_cnt[b], 1);
  }
}

__global__ void k_ie_scatter(FrameDev F) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ns; i += gridDim.x * blockDim.x) {
    const int b = F.ie_bin[i];
    if (b < 0) continue;
    const int pos = F.ie_first[b] + F.ie_slot[i];
    F.ie_idx[pos] = i;
    const float* ie = F.st_ie + (long)i * kStateF;
    F.ie_rec[pos] = make_float4(ie[0], ie[1], ie[20], __int_as_float(i));
  }
}

// n consecutive queue items per calling lane, one atomic per warp.
__device__ __forceinline__ int queue_next_n(int* q, int n) {
  const unsigned mask = __activemask();
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(mask) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(q, __popc(mask) * n);
  base = __shfl_sync(mask, base, leader);
  return base + __popc(mask & ((1u << lane) - 1u)) * n;
}

// chi2 of a 5-vector difference with a Cholesky factorisation (-1: not PD).
__device__ __forceinline__ float chi2_5(const float* d, const float* c) {
  float L[15];  // lower triangle, same indexing as the covariance
  for (int j = 0; j < 5; ++j) {
    float s = c[j * (j + 1) / 2 + j];
    for (int k = 0; k < j; ++k) s = s - L[j * (j + 1) / 2 + k] * L[j * (j + 1) / 2 + k];
    if (!(s > 0.0f)) return -1.0f;
    L[j * (j + 1) / 2 + j] = sqrtf(s);
    for (int i = j + 1; i < 5; ++i) {
      float v = c[i * (i + 1) / 2 + j];
      for (int k = 0; k < j; ++k) v = v - L[i * (i + 1) / 2 + k] * L[j * (j + 1) / 2 + k];
      L[i * (i + 1) / 2 + j] = v / L[j * (j + 1) / 2 + j];
    }
  }
  float yv[5];
  float chi2 = 0.0f;
  for (int i = 0; i < 5; ++i) {
    float v = d[i];
    for (int k = 0; k < i; ++k) v = v - L[i * (i + 1) / 2 + k] * yv[k];
    yv[i] = v / L[i * (i + 1) / 2 + i];
    chi2 = chi2 + yv[i] * yv[i];
  }
  return chi2;
}

// The pair test of the outer end of A against the inner end of B.
__device__ __forceinline__ bool merge_test(const FrameDev& F, const KParams& P, int a, int b,
                                           float& chi2) {
  const int half = P.n_phi;
  const int sa = F.st_sector[a], sb = F.st_sector[b];
  if (sa / half != sb / half) return false;
  const int ds = ((sb % half) - (sa % half) + half) % half;
  if (ds != 0 && ds != 1 && ds != half - 1) return false;
  const int gap = F.st_rmin[b] - F.st_rmax[a];
  if (gap < 1 || gap > P.merge_max_gap) return false;
  const float* oe = F.st_oe + (long)a * kStateF;
  const float* ie = F.st_ie + (long)b * kStateF;
  const float zwin = P.merge_dz + fabsf(oe[3]) * P.merge_zspan;
  if (!(fabsf(ie[1] - oe[1]) <= zwin)) return false;
  Trk<float> t;
  get_state(oe, t);
  if (ds == 1 && !rotate(t, 1, P, P.fit_max_snp)) return false;
  if (ds == half - 1 && !rotate(t, -1, P, P.fit_max_snp)) return false;
  if (!propagate(t, ie[20], P, P.fit_max_snp)) return false;
  float d[5], c[15];
#pragma unroll
  for (int i = 0; i < 5; ++i) d[i] = ie[i] - t.p[i];
  if (!(fabsf(d[0]) <= P.merge_dy) || !(fabsf(d[1]) <= P.merge_dz)) return false;
#pragma unroll
  for (int i = 0; i < 15; ++i) c[i] = t.c[i] + ie[5 + i];
  chi2 = chi2_5(d, c);
  return chi2 >= 0.0f && chi2 < P.merge_chi2;
}

// Position prefilter of the pair test.  A's outer end turned into the frame
// of one of the three sectors searched (q = 0: its own, 1: the next, 2: the
// previous), with the terms of the helix step that depend on A alone; then
// A's position at B's x by the helix step's own expressions for y and z.  The
// prefilter rejects a candidate only where that position lies outside the
// window by more than a rounding margin, and leaves a failed rotation or step
// to the full test, so every decision is the full test's (merge_test), in
// either arithmetic mode.  Nearly all candidates of the index end here,
// before the covariance transport and the 5x5 chi2.
struct MergeA {
  float y, z, s0, c0, kap, tgl, x;
  int ok;
};

__device__ __forceinline__ MergeA merge_a(const float* oe, int q, const KParams& P) {
  Trk<float> t;  // the covariance is not read: its transport is dropped
#pragma unroll
  for (int i = 0; i < 5; ++i) t.p[i] = oe[i];
#pragma unroll
  for (int i = 0; i < 15; ++i) t.c[i] = 0.0f;
  t.x = oe[20];
  bool ok = true;
  if (q == 1) ok = rotate(t, 1, P, P.fit_max_snp);
  else if (q == 2) ok = rotate(t, -1, P, P.fit_max_snp);
  MergeA m;
  m.y = t.p[0];
  m.z = t.p[1];
  m.s0 = t.p[2];
  m.tgl = t.p[3];
  m.kap = t.p[4] * P.kb;
  m.x = t.x;
#ifdef TPC_FAST_ARITH
  const float a0 = 1.0f - m.s0 * m.s0;
  m.c0 = a0 * rsqrtf(a0);
#else
  m.c0 = sqrtf(1.0f - m.s0 * m.s0);
#endif
  m.ok = ok ? 1 : 0;
  return m;
}

// The position (y, z) of A at x = xb (false: no rotation or no step).
__device__ __forceinline__ bool merge_pos(const MergeA& m, float xb, const KParams& P, float& yb,
                                          float& zb) {
  if (!m.ok) return false;
  const float dx = xb - m.x;
  const float s1 = m.s0 + m.kap * dx;
  if (!(fabsf(s1) < P.fit_max_snp)) return false;
#ifdef TPC_FAST_ARITH
  const float a1 = 1.0f - s1 * s1;
  const float c1 = a1 * rsqrtf(a1);
  const float t = (m.s0 + s1) * frcp(m.c0 + c1);
  const float tt = 1.0f + t * t;
  const float L1 = tt * rsqrtf(tt);
#else
  const float c1 = sqrtf(1.0f - s1 * s1);
  const float t = (m.s0 + s1) / (m.c0 + c1);
  const float L1 = sqrtf(1.0f + t * t);
#endif
  const float chord = dx * L1;
  const float u = m.kap * chord * 0.5f;
  yb = m.y + dx * t;
  zb = m.z + m.tgl * (chord * asinc_f(u));
  return true;
}

// z window of the candidates of an outer end in the frame of MergeA m, for
// inner ends on rows with x in [x0, x1].  The full test needs B's z within
// merge_dz of A's z at B's x.  sin(phi) is linear in x, so over the run |sin(phi)|
// stays below its larger end value (and below fit_max_snp, beyond which the
// test fails), and the arc from A to B lies between dx and dx / cos(phi) of that
// value; the arc times tan(lambda) bounds the z step.  0.1 % and 0.02 cm + 1e-5
// |z| cover the rounding of both evaluations.  Against the window the index
// was searched with before (both signs, the steepest angle the cuts allow) it
// is several times shorter, and so are the ranges and candidates to visit.
__device__ __forceinline__ void merge_window(const MergeA& m, float x0, float x1, const KParams& P,
                                             float& zlo, float& zhi) {
  const float d0 = x0 - m.x, d1 = x1 - m.x;
  const float s = fminf(fmaxf(fabsf(m.s0), fmaxf(fabsf(m.s0 + m.kap * d0),
                                                 fabsf(m.s0 + m.kap * d1))),
                        P.fit_max_snp);
  const float rc = 1.001f * rsqrtf(1.0f - s * s);
  const float a0 = d0 < 0.0f ? d0 * rc : d0 * 0.999f;  // shortest (most negative) arc
  const float a1 = d1 > 0.0f ? d1 * rc : d1 * 0.999f;  // longest
  const float e0 = m.tgl * a0, e1 = m.tgl * a1;
  const float mg = P.merge_dz + 0.02f + 1e-5f * (fabsf(m.z) + fabsf(e0) + fabsf(e1));
  zlo = m.z + fminf(e0, e1) - mg;
  zhi = m.z + fmaxf(e0, e1) + mg;
}

// Best merge partner of every outer end A, searched by a group of G lanes
// (G = 1: one thread per end).  The (sector, z bin) ranges of A's candidates
// in the index are dealt out to the lanes, their sizes summed by a group scan,
// and the candidates of all ranges dealt out G at a time; each lane runs the
// pair test of its candidate and the group's smallest (chi2, key of B) is
// found by shuffles.  The minimum does not depend on the visiting order, so
// every G gives the scalar search's result bit for bit.
template <int G>
__global__ void __launch_bounds__(256, 4) k_merge_best(FrameDev F, KParams P) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  const int lane = threadIdx.x & 31;
  const int gl = lane & (G - 1);
  const unsigned gmask = G == 32 ? 0xFFFFFFFFu : (((1u << G) - 1u) << (lane & ~(G - 1)));
  const int half = P.n_phi;
  // up to kFetch ends per queue fetch: lane gl < fetch of the group looks at
  // end base + gl; the ends with no row to search (those that reach the last
  // rows) are answered at once, the others searched one after the other by the
  // whole group.  (A few ends per fetch, so that the atomics stay few; one
  // where the ends are too few to give every group several fetches, as a
  // group's ends are a serial chain.)
  constexpr int kFetch = G < 8 ? G : 8;
  const int groups = (int)(gridDim.x * blockDim.x) / G;
  const int fetch = max(1, min(kFetch, ns / (4 * groups)));
  for (;;) {
    int base = 0;
    if (gl == 0) base = queue_next_n(&F.cnt->queue[kQMerge], fetch);
    base = __shfl_sync(gmask, base, 0, G);
    if (base >= ns) break;
    const int am = base + gl;
    bool live = false;
    // (an outer end linked by the edge following is not searched)
    if (gl < fetch && am < ns && F.st_ok[am] && F.st_next[am] < 0) {
      const int rmx = F.st_rmax[am];
      live = rmx + 1 <= min(rmx + P.merge_max_gap, P.n_rows - 1);
      if (!live) {
        F.st_bestB[am] = -1;
        F.st_bestchi[am] = 0.0f;
      }
    }
    // A's state and z bins in the three sectors searched: lane 3 e + q of the
    // group prepares sector q of the round's e-th end (kSetup ends at once; with
    // fewer than four lanes every lane prepares the three of each end itself) and
    // hands them to the lanes by shuffles; no bins where A cannot be turned into
    // the sector, as the test fails there
    constexpr int kSetup = G >= 4 ? G / 3 : 1;
    for (unsigned todo = __ballot_sync(gmask, live) & gmask; todo;) {
      const int slot = gl / 3;  // the lane's end among the next kSetup
      unsigned mine = todo;
      if (G >= 4)
        for (int e = 0; e < slot && mine; ++e) mine &= mine - 1;
      MergeA ma{};
      int my_s = 0, my_z = 0, my_n = 0;
      const int ae = __shfl_sync(gmask, am, mine ? (__ffs(mine) - 1) & (G - 1) : 0, G);
      auto setup = [&](int a, int q) {
        const float* oe = F.st_oe + (long)a * kStateF;
        const int sa = F.st_sector[a], rmx = F.st_rmax[a];
        const float zwin = P.merge_dz + fabsf(oe[3]) * P.merge_zspan;
        ma = merge_a(oe, q, P);
        my_s = sa / half * half + (sa % half + (q == 0 ? 0 : q == 1 ? 1 : half - 1)) % half;
        float zlo, zhi;
        merge_window(ma, F.row_x[rmx + 1], F.row_x[min(rmx + P.merge_max_gap, P.n_rows - 1)], P,
                     zlo, zhi);
        zlo = fmaxf(zlo, oe[1] - zwin - 0.01f);
        zhi = fminf(zhi, oe[1] + zwin + 0.01f);
        my_z = merge_zbin(F, my_s, zlo);
        my_n = ma.ok && zlo <= zhi ? merge_zbin(F, my_s, zhi) - my_z + 1 : 0;
      };
      if (G >= 4 && slot < kSetup && mine) setup(ae, gl - 3 * slot);
#pragma unroll 1
      for (int e = 0; e < kSetup && todo; ++e, todo &= todo - 1) {
        const int a = __shfl_sync(gmask, am, (__ffs(todo) - 1) & (G - 1), G);
        const int keyA = F.st_key[a];
        unsigned long long best = ~0ull;
        int bb = -1;
        // the pair test needs 1 <= rmin(B) - rmax(A) <= merge_max_gap: only
        // those rows of the index are visited
        const int r0 = F.st_rmax[a] + 1;
        const int r1 = min(F.st_rmax[a] + P.merge_max_gap, P.n_rows - 1);
        const float* oe = F.st_oe + (long)a * kStateF;
        const float zwin = P.merge_dz + fabsf(oe[3]) * P.merge_zspan;
        const float oz = oe[1];
        int sq[3], zq[3], nq[3];
        int nr = 0;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          if (G < 4) {
            setup(a, q);
            sq[q] = my_s;
            zq[q] = my_z;
            nq[q] = my_n;
          } else {
            sq[q] = __shfl_sync(gmask, my_s, 3 * e + q, G);
            zq[q] = __shfl_sync(gmask, my_z, 3 * e + q, G);
            nq[q] = __shfl_sync(gmask, my_n, 3 * e + q, G);
          }
          nr += nq[q];
        }
        for (int j0 = 0; j0 < nr; j0 += G) {
          int lo = 0, cnt = 0, qj = 0;
          int j = j0 + gl;
          if (j < nr) {
            const int q = j < nq[0] ? 0 : j < nq[0] + nq[1] ? 1 : 2;
            j -= q == 0 ? 0 : q == 1 ? nq[0] : nq[0] + nq[1];
            const int base = ((q == 0 ? sq[0] : q == 1 ? sq[1] : sq[2]) * kMergeZ +
                              (q == 0 ? zq[0] : q == 1 ? zq[1] : zq[2]) + j) * P.n_rows;
            lo = F.ie_first[base + r0];
            cnt = F.ie_first[base + r1 + 1] - lo;
            qj = q;
          }
          int inc = cnt;  // inclusive scan of the range sizes over the group
#pragma unroll
          for (int o = 1; o < G; o <<= 1) {
            const int v = __shfl_up_sync(gmask, inc, o, G);
            if (gl >= o) inc += v;
          }
          const int total = __shfl_sync(gmask, inc, G - 1, G);
          for (int c0 = 0; c0 < total; c0 += G) {
            const int c = c0 + gl;
            int L = 0;  // the range holding candidate c: first lane with inc > c
#pragma unroll
            for (int st = G / 2; st >= 1; st >>= 1) {
              const int v = __shfl_sync(gmask, inc, L + st - 1, G);
              if (v <= c) L += st;
            }
            const int excl = __shfl_sync(gmask, inc - cnt, L, G);
            const int lo_l = __shfl_sync(gmask, lo, L, G);
            const int q_l = __shfl_sync(gmask, qj, L, G);
            MergeA mq;
            if (G >= 4) {
              mq.y = __shfl_sync(gmask, ma.y, 3 * e + q_l, G);
              mq.z = __shfl_sync(gmask, ma.z, 3 * e + q_l, G);
              mq.s0 = __shfl_sync(gmask, ma.s0, 3 * e + q_l, G);
              mq.c0 = __shfl_sync(gmask, ma.c0, 3 * e + q_l, G);
              mq.kap = __shfl_sync(gmask, ma.kap, 3 * e + q_l, G);
              mq.tgl = __shfl_sync(gmask, ma.tgl, 3 * e + q_l, G);
              mq.x = __shfl_sync(gmask, ma.x, 3 * e + q_l, G);
              mq.ok = __shfl_sync(gmask, ma.ok, 3 * e + q_l, G);
            }
            if (c >= total) continue;
            // the indexed inner end: (y, z, x, track)
            const float4 rec = F.ie_rec[lo_l + (c - excl)];
            if (!(fabsf(rec.y - oz) <= zwin)) continue;  // the full test's z window
            if (G < 4) mq = merge_a(oe, q_l, P);
            float yb, zb;
            if (merge_pos(mq, rec.z, P, yb, zb) &&
                (fabsf(rec.x - yb) > P.merge_dy + 0.01f + 1e-5f * fabsf(rec.x) ||
                 fabsf(rec.y - zb) > P.merge_dz + 0.01f + 1e-5f * fabsf(rec.y)))
              continue;
            const int b = __float_as_int(rec.w);
            if (b == a || !F.st_ok[b]) continue;
            float chi2;
            if (!merge_test(F, P, a, b, chi2)) continue;
            const unsigned long long kb = pack_chi_key(chi2, F.st_key[b]);
            if (kb < best) {
              best = kb;
              bb = b;
            }
            atomicMin(&F.st_bestA[b], pack_chi_key(chi2, keyA));
          }
        }
#pragma unroll
        for (int o = G / 2; o >= 1; o >>= 1) {
          const unsigned long long ob = __shfl_xor_sync(gmask, best, o, G);
          const int obb = __shfl_xor_sync(gmask, bb, o, G);
          if (ob < best) {
            best = ob;
            bb = obb;
          }
        }
        if (gl == 0) {
          F.st_bestB[a] = bb;
          F.st_bestchi[a] = bb >= 0 ? o2f((unsigned)(best >> 32)) : 0.0f;
        }
      }
    }
  }
}

__global__ void k_merge_link(FrameDev F) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < ns; a += gridDim.x * blockDim.x) {
    const int b = F.st_bestB[a];
    if (b < 0) continue;
    if (F.st_bestA[b] == pack_chi_key(F.st_bestchi[a], F.st_key[a])) {
      F.st_next[a] = b;
      F.st_hasprev[b] = 1;
    }
  }
}

// ------------------------------------------ across the central electrode
// chi2 of the 4-vector (y, sin phi, tan lambda, q/pT) of a 5-vector difference
// with the marginal covariance (z left out).
__device__ __forceinline__ float chi2_4z(const float* d, const float* c) {
  const int ix[4] = {0, 2, 3, 4};
  float L[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float sj = c[ix[j] * (ix[j] + 1) / 2 + ix[j]];
    for (int k = 0; k < j; ++k) sj = sj - L[j][k] * L[j][k];
    if (!(sj > 0.0f)) return -1.0f;
    L[j][j] = sqrtf(sj);
    for (int i = j + 1; i < 4; ++i) {
      float v = c[ix[i] * (ix[i] + 1) / 2 + ix[j]];
      for (int k = 0; k < j; ++k) v = v - L[i][k] * L[j][k];
      L[i][j] = v / L[j][j];
    }
  }
  float yv[4];
  float chi2 = 0.0f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float v = d[ix[i]];
    for (int k = 0; k < i; ++k) v = v - L[i][k] * yv[k];
    yv[i] = v / L[i][i];
    chi2 = chi2 + yv[i] * yv[i];
  }
  return chi2;
}

// Pair test across the central electrode (Sec. 2 merges "then across the
// central electrode"): the outer end of A and the inner end of B in the same
// azimuthal sector of one frame on the two sides, B's innermost row 1 to
// merge_max_gap rows above A's outermost.  The measured z of the two sides
// differ by 2 vd t0 with t0 unknown in continuous readout (Sec. 1): z stays out
// of the chi2 (4 dof, summed covariances, below merge_chi2), and the sum of
// the two ends' z, in which t0 cancels, must lie within twice merge_dz +
// |tan lambda| * merge_zspan.  dz = z_A - z_B at B's x is the shift that
// brings B's side into A's measured z.
__device__ __forceinline__ bool cross_test(const FrameDev& F, const KParams& P, int a, int b,
                                           float& chi2, float& dz) {
  const int half = P.n_phi;
  const int sa = F.st_sector[a], sb = F.st_sector[b];
  if (sa / (2 * half) != sb / (2 * half) || sa / half == sb / half || sa % half != sb % half)
    return false;
  const int gap = F.st_rmin[b] - F.st_rmax[a];
  if (gap < 1 || gap > P.merge_max_gap) return false;
  const float* oe = F.st_oe + (long)a * kStateF;
  const float* ie = F.st_ie + (long)b * kStateF;
  const float zwin = P.merge_dz + fabsf(oe[3]) * P.merge_zspan;
  if (!(fabsf(oe[1] + ie[1]) <= zwin + zwin)) return false;
  Trk<float> t;
  get_state(oe, t);
  if (!propagate(t, ie[20], P, P.fit_max_snp)) return false;
  float d[5], c[15];
#pragma unroll
  for (int i = 0; i < 5; ++i) d[i] = ie[i] - t.p[i];
  if (!(fabsf(d[0]) <= P.merge_dy)) return false;
#pragma unroll
  for (int i = 0; i < 15; ++i) c[i] = t.c[i] + ie[5 + i];
  chi2 = chi2_4z(d, c);
  dz = t.p[1] - ie[1];
  return chi2 >= 0.0f && chi2 < P.merge_chi2;
}

// Chain ends against chain starts of the other side (after the merging within
// each side): the best start of every end; each start keeps its best end.
__global__ void k_cross_best(FrameDev F, KParams P) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  const int half = P.n_phi;
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < ns; a += gridDim.x * blockDim.x) {
    if (!F.st_ok[a] || F.st_next[a] >= 0) continue;
    const int keyA = F.st_key[a];
    const int sa = F.st_sector[a];
    const int base = sa - sa % (2 * half);
    const int sb = base + (sa % (2 * half) + half) % (2 * half);
    const float* oe = F.st_oe + (long)a * kStateF;
    const float zwin = P.merge_dz + fabsf(oe[3]) * P.merge_zspan;
    const int r0 = F.st_rmax[a] + 1;
    const int r1 = min(F.st_rmax[a] + P.merge_max_gap, P.n_rows - 1);
    if (r0 > r1) continue;
    // the test needs |z_A + z_B| <= 2 zwin: B's inner-end z around -z_A
    const float m = 0.01f;
    const int z0 = merge_zbin(F, sb, -oe[1] - 2.0f * zwin - m);
    const int z1 = merge_zbin(F, sb, -oe[1] + 2.0f * zwin + m);
    int bb = -1, bkey = 0;
    float bchi = 0.0f, bdz = 0.0f;
    for (int zb = z0; zb <= z1; ++zb) {
      const int bin0 = (sb * kMergeZ + zb) * P.n_rows;
      const int lo = F.ie_first[bin0 + r0], hi = F.ie_first[bin0 + r1 + 1];
      for (int k = lo; k < hi; ++k) {
        const int b = F.ie_idx[k];
        if (!F.st_ok[b] || F.st_hasprev[b]) continue;
        float chi2, dz;
        if (!cross_test(F, P, a, b, chi2, dz)) continue;
        const int kb = F.st_key[b];
        if (bb < 0 || chi2 < bchi || (chi2 == bchi && kb < bkey)) {
          bb = b;
          bchi = chi2;
          bkey = kb;
          bdz = dz;
        }
        atomicMin(&F.st_xbestA[b], pack_chi_key(chi2, keyA));
      }
    }
    F.st_xbestB[a] = bb;
    F.st_xchi[a] = bchi;
    F.st_xdz[a] = bdz;
  }
}

__global__ void k_cross_link(FrameDev F) {
  const int ns = F.cnt->n_tracks;
  if (F.cnt->err) return;
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < ns; a += gridDim.x * blockDim.x) {
    const int b = F.st_xbestB[a];
    if (b < 0) continue;
    if (F.st_xbestA[b] == pack_chi_key(F.st_xchi[a], F.st_key[a])) {
      F.st_next[a] = b;
      F.st_hasprev[b] = 1;
      F.st_dz[b] = F.st_xdz[a];
    }
  }
}

// Heads of chains -> fit tracks (compaction in sector-track order).
__device__ __forceinline__ int is_head(const FrameDev& F, int i, int ns) {
  return (i < ns && F.st_ok[i] && !F.st_hasprev[i]) ? 1 : 0;
}

__global__ void k_head_count(FrameDev F) {
  __shared__ int sh[32];
  const int ns = F.cnt->n_tracks;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int f = F.cnt->err ? 0 : is_head(F, i, ns);
  int tot;
  block_exscan(f, sh, &tot);
  if (threadIdx.x == 0) F.scan_tmp[blockIdx.x] = tot;
}

// Head list, plus whether the chain's fit updates run in FP64 (|q/pT| at
// its inner end above looper_qpt).
__global__ void k_head_write(FrameDev F, KParams P) {
  __shared__ int sh[32];
  const int ns = F.cnt->n_tracks;
  if (blockIdx.x == 0 && threadIdx.x == 0 && F.cnt->n_merged > F.cap_ft) {
    atomicOr(&F.cnt->err, kErrCapTracks);
    atomicMax(&F.cnt->need_tracks, F.cnt->n_merged);
  }
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int f = F.cnt->err ? 0 : is_head(F, i, ns);
  int tot;
  const int ex = block_exscan(f, sh, &tot);
  const int pos = F.scan_tmp[blockIdx.x] + ex;
  if (f && pos < F.cap_ft) {
    F.ft_head[pos] = i;
    const float q = fabsf(F.st_ie[(long)i * kStateF + 4]);
    F.ft_looper[pos] = (P.looper_qpt > 0.0f && q > P.looper_qpt) ? 1 : 0;
  }
}

// Processing order of the fit kernels: a stable partition of the fit tracks,
// loopers first.  A looper's update costs its whole warp about twice the other
// update's time, so loopers share warps, and the longer work starts first; each
// part keeps list order (sector-major) but for the order by stations within a
// stretch (k_fit_order), which keeps the cluster accesses of a warp close
// together.  No result depends on the order.
__device__ __forceinline__ int looper_flag(const FrameDev& F, int f) {
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  return (!F.cnt->err && f < nf) ? F.ft_looper[f] : 0;
}

__global__ void k_looper_count(FrameDev F) {
  __shared__ int sh[32];
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  int tot;
  block_exscan(looper_flag(F, f), sh, &tot);
  if (threadIdx.x == 0) F.scan_tmp[blockIdx.x] = tot;
}

__global__ void k_looper_write(FrameDev F) {
  __shared__ int sh[32];
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  const int fl = looper_flag(F, f);
  int tot;
  const int lr = F.scan_tmp[blockIdx.x] + block_exscan(fl, sh, &tot);  // loopers before f
  if (F.cnt->err || f >= nf) return;
  F.ft_order[fl ? lr : F.cnt->n_loopers + (f - lr)] = f;
}

// The fit kernels take ft_order: loopers in [0, nL), the other tracks in [nL, nf),
// which are numbered from the next multiple of 32 on, so that no warp starts
// with both kinds (on a frame of a few dozen tracks every warp would, and pay for
// both updates in each step).  All in one launch per iteration: iteration 3 in
// two, the other tracks in 80 registers first, took 0.78 against 0.61 ms on two
// full frames and 0.24 against 0.17 on a central event.
__device__ __forceinline__ int fit_total(int nL, int nf) { return nf + ((32 - (nL & 31)) & 31); }
__device__ __forceinline__ int fit_position(int q, int nL) {  // -1: no track
  const int pad = (32 - (nL & 31)) & 31;
  return q < nL ? q : q < nL + pad ? -1 : q - pad;
}

// ------------------------------------------ a9/a10 linearised three-iteration fit
struct Lin {
  Trk<float> t;
  float r[5];
  int sector;
};

__device__ __forceinline__ void lin_start(Lin& L, const Trk<float>& s, int sector,
                                          const KParams& P) {
  L.t = s;
  reset_cov(L.t.c, P);
#pragma unroll
  for (int i = 0; i < 5; ++i) L.r[i] = s.p[i];
  L.sector = sector;
}

__device__ __forceinline__ bool lin_rotate(Lin& L, int dir, const KParams& P,
                                           float* jrec = nullptr) {
  const float ca = P.rot_c;
  const float sa = dir > 0 ? P.rot_s : -P.rot_s;
  const float snp = L.r[2];
  const float csp = sqrtf(1.0f - snp * snp);
  const float xn = L.t.x * ca + L.r[0] * sa;
  const float yn = L.r[0] * ca - L.t.x * sa;
  const float sn = snp * ca - csp * sa;
  const float cn = csp * ca + snp * sa;
  if (!(cn > 0.0f) || !(fabsf(sn) < P.fit_max_snp)) return false;
  const float j00 = csp / cn;
  const float j10 = -sa * L.r[3] / cn;
  const float j20 = -sa * (L.r[4] * P.kb);
  const float j22 = cn / csp;
  const float d0 = L.t.p[0] - L.r[0], d1 = L.t.p[1] - L.r[1], d2 = L.t.p[2] - L.r[2];
  float* c = L.t.c;
  const float m00 = c[0], m10 = c[1], m11 = c[2], m20 = c[3], m21 = c[4], m22 = c[5];
  const float m30 = c[6], m31 = c[7], m32 = c[8], m33 = c[9];
  const float m40 = c[10], m41 = c[11], m42 = c[12], m43 = c[13], m44 = c[14];
  const float a00 = j00 * m00;
  const float a10 = j10 * m00 + m10, a11 = j10 * m10 + m11;
  const float a20 = j20 * m00 + j22 * m20, a21 = j20 * m10 + j22 * m21,
              a22 = j20 * m20 + j22 * m22;
  c[0] = a00 * j00;
  c[1] = a10 * j00;
  c[2] = a10 * j10 + a11;
  c[3] = a20 * j00;
  c[4] = a20 * j10 + a21;
  c[5] = a20 * j20 + a22 * j22;
  c[6] = m30 * j00;
  c[7] = m30 * j10 + m31;
  c[8] = m30 * j20 + m32 * j22;
  c[9] = m33;
  c[10] = m40 * j00;
  c[11] = m40 * j10 + m41;
  c[12] = m40 * j20 + m42 * j22;
  c[13] = m43;
  c[14] = m44;
  L.r[0] = yn;
  L.r[2] = sn;
  L.t.x = xn;
  L.t.p[0] = L.r[0] + j00 * d0;
  L.t.p[1] = L.r[1] + (j10 * d0 + d1);
  L.t.p[2] = L.r[2] + (j20 * d0 + j22 * d2);
  if (jrec) {
    jrec[0] = j00;
    jrec[1] = j10;
    jrec[2] = j20;
    jrec[3] = j22;
  }
  return true;
}

__device__ __forceinline__ bool lin_propagate(Lin& L, float xnew, const KParams& P,
                                              StepJ* frec = nullptr) {
  const float dx = xnew - L.t.x;
  StepJ st;
  if (!helix_step(L.r, dx, P, st, P.fit_max_snp)) return false;
  if (frec) *frec = st;
  const float d0 = L.t.p[0] - L.r[0], d1 = L.t.p[1] - L.r[1], d2 = L.t.p[2] - L.r[2];
  const float d3 = L.t.p[3] - L.r[3], d4 = L.t.p[4] - L.r[4];
  L.r[0] = st.p0;
  L.r[1] = st.p1;
  L.r[2] = st.p2;
  L.t.p[0] = L.r[0] + (d0 + st.f02 * d2 + st.f04 * d4);
  L.t.p[1] = L.r[1] + (d1 + st.f12 * d2 + st.f13 * d3 + st.f14 * d4);
  L.t.p[2] = L.r[2] + (d2 + st.f24 * d4);
  cov_transport(L.t.c, st);
  add_ms(L.t.c, L.r, dx, P);
  L.t.x = xnew;
  return true;
}

// Station change: rotation (when the sector changes) and propagation.  The
// optional records receive the rotation Jacobian (jrec, untouched without a
// rotation) and the propagation Jacobian (frec) for the adjoint.
__device__ __forceinline__ bool lin_goto(Lin& L, int sector, float x, const KParams& P,
                                         float* jrec = nullptr, StepJ* frec = nullptr) {
  if (sector != L.sector) {
    const int half = P.n_phi;
    const int ds = ((sector % half) - (L.sector % half) + half) % half;
    if (ds == 1) {
      if (!lin_rotate(L, 1, P, jrec)) return false;
    } else if (ds == half - 1) {
      if (!lin_rotate(L, -1, P, jrec)) return false;
    } else if (ds != 0) {
      return false;
    }
    // ds == 0: the same azimuthal sector on the other side of the central
    // electrode, whose local frame is the same
    L.sector = sector;
  }
  return lin_propagate(L, x, P, frec);
}

__device__ __forceinline__ void inv2(float a00, float a01, float a11, float& i00, float& i01,
                                     float& i11) {
  const float idet = frcp(a00 * a11 - a01 * a01);
  i00 = a11 * idet;
  i01 = -a01 * idet;
  i11 = a00 * idet;
}

struct Interp {
  float y, z, c00, c01, c11;
};

__device__ __forceinline__ Interp interpolate(const float* a, const float* b) {
  float wa00, wa01, wa11, wb00, wb01, wb11;
  inv2(a[2], a[3], a[4], wa00, wa01, wa11);
  inv2(b[2], b[3], b[4], wb00, wb01, wb11);
  Interp I;
  inv2(wa00 + wb00, wa01 + wb01, wa11 + wb11, I.c00, I.c01, I.c11);
  const float v0 = (wa00 * a[0] + wa01 * a[1]) + (wb00 * b[0] + wb01 * b[1]);
  const float v1 = (wa01 * a[0] + wa11 * a[1]) + (wb01 * b[0] + wb11 * b[1]);
  I.y = I.c00 * v0 + I.c01 * v1;
  I.z = I.c01 * v0 + I.c11 * v1;
  return I;
}

__device__ __forceinline__ float chi2_interp(const Interp& I, float my, float mz,
                                             const KParams& P) {
  // (explicitly rounded: fused with the products they come from or not, as the
  // compiler finds them in one basic block or in two, these would let the cut's
  // decision depend on the kernel that evaluates it)
  float w00, w01, w11;
  inv2(__fadd_rn(I.c00, P.sy2), I.c01, __fadd_rn(I.c11, P.sz2), w00, w01, w11);
  const float r0 = __fsub_rn(my, I.y), r1 = __fsub_rn(mz, I.z);
  return r0 * (w00 * r0 + w01 * r1) + r1 * (w01 * r0 + w11 * r1);
}

// Station list of fit track f: clusters of the chain (rows increasing) plus
// empty inner rows between two clusters of one sector.
__device__ __forceinline__ float zoff(const float* ie) {
  return ie[1] - ie[3] * sqrtf(ie[20] * ie[20] + ie[0] * ie[0]);
}

// Tracks merged across the central electrode: the measured z of a cluster of
// sector sec in the frame of the track's first side (zside: the side whose
// clusters take the shift zsh, -1 for a track on one side), and the window
// centre cz of that frame in the measured z of sector sec.
__device__ __forceinline__ int shift_side(const FrameDev& F, int f) {
  return F.ft_zsh[f] != 0.0f ? 1 - F.ft_side0[f] : -1;
}
__device__ __forceinline__ float track_z(float z, int sec, int zside, float zsh, const KParams& P) {
  return zside >= 0 && ((sec / P.n_phi) & 1) == zside ? z + zsh : z;
}
// The shift that applies to the clusters of sector sec (0: none).
__device__ __forceinline__ float row_shift(int sec, int zside, float zsh, const KParams& P) {
  return zside >= 0 && ((sec / P.n_phi) & 1) == zside ? zsh : 0.0f;
}

// A station's measurement for the fit iterations: the cluster's position in
// the frame of the track's first side, corrected by the map, with the map's x
// displacement apart (it moves the cluster along the reference of the
// iteration that uses it).  The correction depends on the row's x, the cluster
// and the track's z offset, not on the filter state, so it is evaluated once
// per station here, over all stations at once, instead of in each iteration on
// its serial chain of steps.
template <bool kMap>
__device__ __forceinline__ float4 fit_meas(const MapDev& M, const KParams& P, int rs, float x,
                                           float y, float z, float z0) {
  const int sec = rs / P.n_rows, row = rs % P.n_rows;
  float4 m = make_float4(0.0f, y, z, __uint_as_float((unsigned)sec << 8 | (unsigned)row | kStHave));
  if (kMap) {
    float D[3];
    map_eval(M, P, sec, x, y, z - z0, D);
    m.x = D[0];
    m.y = y + D[1];
    m.z = z + D[2];
  }
  return m;
}

// The measurement (my, mz) of station record m about the reference ref (false:
// the reference cannot be stepped to the displaced cluster).
template <bool kMap>
__device__ __forceinline__ bool meas_at(const float4& m, const KParams& P, const float* ref,
                                        float& my, float& mz) {
  my = m.y;
  mz = m.z;
  if (kMap && m.x != 0.0f) {
    StepJ st;
    if (!helix_step(ref, m.x, P, st, P.fit_max_snp)) return false;
    my = my - (st.p0 - ref[0]);
    mz = mz - (st.p1 - ref[1]);
  }
  return true;
}

__device__ __forceinline__ int st_row(const float4& m) { return __float_as_int(m.w) & 0xFF; }
__device__ __forceinline__ int st_sector(const float4& m) {
  return (__float_as_int(m.w) >> 8) & 0xFFFF;
}
__device__ __forceinline__ bool st_have(const float4& m) {
  return (__float_as_uint(m.w) & kStHave) != 0u;
}

// Per fit track, ahead of the fit: the station list with the stations'
// measurements, the chain's last segment (whose outer end starts iteration 1),
// the identity key and the drift-time z offset.  A station is a kept cluster,
// preceded, on the inner rows of one sector, by an empty station on every row
// skipped since the previous cluster.  Stations beyond kMaxRows are dropped
// (none are reached: a chain's rows increase along it).
//
// A warp takes 32 tracks.  Its lanes walk their tracks' chains side by side,
// one segment per round, so that the dependent loads of a segment's header
// (next segment, tracklet, length, position offset) are in flight for 32 tracks
// at once; then the warp writes the round's segments one after the other, its
// lanes over 32 kept clusters at a time (their positions lie in one run, from
// the sector refit's gather), a warp scan of the stations each cluster adds
// giving the places.
template <bool kMap>
__global__ void __launch_bounds__(kBlock, 3) k_fit_stations(FrameDev F, KParams P, MapDev M) {
  if (!kMap) M.on = 0;
  __shared__ float rx[kMaxRows];
  for (int r = threadIdx.x; r < P.n_rows; r += blockDim.x) rx[r] = F.row_x[r];
  __syncthreads();
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  const int NR = P.n_rows;
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (blockDim.x >> 5);
  const int per = warp_share(nf, nw);
  for (int f0 = per * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); f0 < nf;
       f0 += per * nw) {
    const int f = f0 + lane;
    const bool mine = lane < per && f < nf;
    const int head = mine ? F.ft_head[f] : -1;
    // across the central electrode: the side of the first segment, and the
    // z shift of the clusters on the other side (set at the first segment
    // there, 0 for a chain on one side)
    const int side0 = mine ? (F.st_sector[head] / P.n_phi) & 1 : 0;
    const float z0 = mine ? zoff(F.st_ie + (long)head * kStateF) : 0.0f;
    float zsh = 0.0f;
    bool crossed = false;
    int sg = head, last = head, ns = 0, prev = -1;
    while (__any_sync(0xffffffffu, sg >= 0)) {
      int ti = 0, nk = 0, off = 0, nxt = -1;
      if (sg >= 0) {
        last = sg;
        nxt = F.st_next[sg];
        off = F.st_off[sg];
        ti = F.st_tl[sg];
        nk = F.tl_nkept[ti];
        if (!crossed && ((F.st_sector[sg] / P.n_phi) & 1) != side0) {
          crossed = true;
          zsh = F.st_dz[sg];
        }
      }
      for (unsigned todo = __ballot_sync(0xffffffffu, sg >= 0); todo; todo &= todo - 1) {
        const int j = __ffs(todo) - 1;
        const int tj = __shfl_sync(0xffffffffu, ti, j);
        const int nj = __shfl_sync(0xffffffffu, nk, j);
        const int oj = __shfl_sync(0xffffffffu, off, j);
        const int sj = __shfl_sync(0xffffffffu, side0, j);
        const float z0j = __shfl_sync(0xffffffffu, z0, j);
        const float zshj = __shfl_sync(0xffffffffu, zsh, j);
        int nsj = __shfl_sync(0xffffffffu, ns, j);
        int pj = __shfl_sync(0xffffffffu, prev, j);
        const int zside = zshj != 0.0f ? 1 - sj : -1;
        const int* K = F.tl_kept + (long)tj * kMaxRows;  // outermost first
        int* SC = F.ft_st_cl + (long)(f0 + j) * kMaxRows;
        uint16_t* SR = F.ft_st_rs + (long)(f0 + j) * kMaxRows;
        float4* SM = F.ft_meas + (long)(f0 + j) * kMaxRows;
        for (int j0 = 0; j0 < nj; j0 += 32) {
          const bool valid = j0 + lane < nj;
          const int q = nj - 1 - (j0 + lane);
          const int c = valid ? K[q] : -1;
          float4 ps = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
          if (valid) {
            if (oj >= 0) {
              ps = F.st_pos[oj + q];
            } else {  // a segment of the edge following
              const float2 yz = F.syz[c];
              const int r = F.srow[c];
              ps = make_float4(rx[r % NR], yz.x, yz.y, __int_as_float(r));
            }
          }
          const int rs = __float_as_int(ps.w);
          int prs = __shfl_up_sync(0xffffffffu, rs, 1);
          if (lane == 0) prs = pj;
          int gap = 0;
          if (valid && prs >= 0 && prs / NR == rs / NR)
            gap = max(0, min(rs % NR, P.inner_rows) - (prs % NR + 1));
          const int add = valid ? gap + 1 : 0;
          int incl = add;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const int v = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += v;
          }
          const int at = nsj + incl - add;
          if (valid) {
            for (int e = 0; e < gap && at + e < kMaxRows; ++e) {
              const int re = rs - rs % NR + prs % NR + 1 + e;
              SC[at + e] = -1;
              SR[at + e] = (uint16_t)re;
              SM[at + e] = make_float4(0.0f, 0.0f, 0.0f,
                                       __uint_as_float((unsigned)(re / NR) << 8 |
                                                       (unsigned)(re % NR)));
            }
            if (at + gap < kMaxRows) {
              SC[at + gap] = c;
              SR[at + gap] = (uint16_t)rs;
              SM[at + gap] = fit_meas<kMap>(M, P, rs, ps.x, ps.y,
                                            track_z(ps.z, rs / NR, zside, zshj, P), z0j);
              // Phase III: clusters held by a station outside the inner region
              // are not extrapolation candidates of any track
              if (P.ext_rows > 0 && rs % NR >= P.inner_rows) F.ft_fixed[c] = 1;
            }
          }
          const int nvalid = min(32, nj - j0);
          nsj += __shfl_sync(0xffffffffu, incl, 31);
          pj = __shfl_sync(0xffffffffu, rs, nvalid - 1);
        }
        if (lane == j) {
          ns = nsj;
          prev = pj;
        }
      }
      sg = nxt;
    }
    if (mine) {
      F.ft_side0[f] = side0;
      F.ft_zsh[f] = zsh;
      F.ft_nst[f] = min(ns, kMaxRows);
      F.ft_key[f] = F.st_key[head];
      F.ft_last[f] = last;
      F.ft_z0[f] = z0;
      F.ft_next[f] = 0;
      F.ft_nout[f] = 0;
    }
  }
}

// The fit tracks' order, stretch by stretch by stations (loopers stay first).
__global__ void __launch_bounds__(kBlock) k_fit_order(FrameDev F) {
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  constexpr int kHalf = kOrdBuckets / 2;
  for (int c0 = blockIdx.x * kOrdChunk; c0 < nf; c0 += gridDim.x * kOrdChunk)
    order_chunk(
        min(kOrdChunk, nf - c0), [&](int q) { return F.ft_order[c0 + q]; },
        [&](int f) {
          return (F.ft_looper[f] ? kHalf - 1 : -1) + min(kHalf - 1, F.ft_nst[f] * kHalf / kMaxRows);
        },
        F.ft_order + c0);
}

// Iterations 1 and 2 of the final fit (k_fit1, k_fit2) run as per-lane state
// machines: every loop iteration is one station (station change, then the
// iteration's own work, then the update) of the lane's current track, and a
// lane whose track ends takes the next one from the work queue, so the lanes
// of a warp issue the update (FP64 for loopers) together however unequal
// their tracks are.  Iteration 1 runs inward storing the predictions;
// iteration 2 runs outward, interpolates with them, flags outliers and
// collects the inner-row candidates (Sec. 3).  Two kernels rather than one:
// each carries only its own iteration's code and registers.
enum : int { kFitIdle = 0, kFitIn, kFitExt };

// One row step of the Phase III extrapolation, also over sector boundaries
// (Sec. 3): to row r in sector sec; beyond the sector's edge there (|y| >
// x tan 10 deg) the track continues in the neighbouring sector of the same
// side on that edge (rotation, then the row's x in the new frame), and stops
// if it still lies beyond that sector's edge plus edge_margin.
__device__ __forceinline__ bool ext_step(Lin& L, int& sec, int r, const float* rx,
                                         const KParams& P) {
  if (!lin_goto(L, sec, rx[r], P)) return false;
  if (fabsf(L.t.p[0]) > L.t.x * P.tan_half) {
    const int half = P.n_phi;
    const int base = sec - sec % half;
    const int nsec = base + (sec % half + (L.t.p[0] > 0.0f ? 1 : half - 1)) % half;
    if (!lin_goto(L, nsec, rx[r], P)) return false;
    sec = nsec;
  }
  return !(fabsf(L.t.p[0]) > L.t.x * P.tan_half + P.edge_margin);
}

__device__ __forceinline__ void inner_candidates(FrameDev& F, const KParams& P, const MapDev& M,
                                                 int f, int k, int rs, float x, const float* ref,
                                                 const Interp& I, float z0, float zadd) {
  const int sec = rs / P.n_rows;
  float cy = I.y, cz = I.z;
  {
    float D[3];
    map_eval(M, P, sec, x, I.y, I.z - z0, D);
    float sy = D[1], sz = D[2];
    if (D[0] != 0.0f) {
      StepJ stp;
      if (helix_step(ref, D[0], P, stp, P.fit_max_snp)) {
        sy = sy - (stp.p0 - ref[0]);
        sz = sz - (stp.p1 - ref[1]);
      }
    }
    cy = I.y - sy;
    cz = I.z - sz;
  }
  const float wy = sqrtf(P.int_chi2 * (I.c00 + P.sy2)) * 1.001f + P.attach_margin;
  const float wz = sqrtf(P.int_chi2 * (I.c11 + P.sz2)) * 1.001f + P.attach_margin;
  if (zadd != 0.0f) cz = cz - zadd;  // the row's measured z
  int* cand = F.ft_cand + ((long)f * F.nslot + k) * kMaxCand;
  float* cchi = F.ft_cchi + ((long)f * F.nslot + k) * kMaxCand;
  int nc = 0;
  int cid[kMaxCand];
  const RowGrid g = F.rows[rs];
  for_window(F.bin_first, g, cy - wy - 0.01f, cy + wy + 0.01f, cz - wz - 0.01f, cz + wz + 0.01f,
             [&](int kk) {
    const float2 pk = F.syz[kk];
    const float yk = pk.x, zk = pk.y;
    if (!(fabsf(yk - cy) <= wy && fabsf(zk - cz) <= wz)) return;
    float my, mz;
    if (!corrected(M, P, sec, x, yk, zadd != 0.0f ? zk + zadd : zk, z0, ref, my, mz)) return;
    const float c2 = chi2_interp(I, my, mz, P);
    if (!(c2 < P.int_chi2)) return;
    const int id = F.sid[kk];
    // insertion into the sorted top-cand_k list by (chi2, id)
    int pos = nc;
    while (pos > 0 && (c2 < cchi[pos - 1] || (c2 == cchi[pos - 1] && id < cid[pos - 1]))) --pos;
    if (pos >= P.cand_k) return;
    const int lim = nc < P.cand_k ? nc : P.cand_k - 1;
    for (int j = lim; j > pos; --j) {
      cand[j] = cand[j - 1];
      cchi[j] = cchi[j - 1];
      cid[j] = cid[j - 1];
    }
    cand[pos] = kk;
    cchi[pos] = c2;
    cid[pos] = id;
    if (nc < P.cand_k) ++nc;
  });
  F.ft_ncand[(long)f * F.nslot + k] = (uint8_t)nc;
  F.ft_assigned[(long)f * F.nslot + k] = -1;
}

// Phase III (Sec. 3): candidates of an extrapolated row (sorted (sector, row)
// rr) into candidate slot `js` of track f -- every cluster not held by a
// station outside the inner region whose chi2 to the prediction is below
// ext_chi2, the best cand_k by (chi2, id), for the second ambiguity solving.
__device__ __forceinline__ void ext_candidates(FrameDev& F, const KParams& P, const MapDev& M, int f,
                                            int js, int rr, const Lin& L, float z0,
                                            float zadd) {
  const int sec = rr / P.n_rows;
  float cy, cz;
  {
    float D[3];
    map_eval(M, P, sec, L.t.x, L.t.p[0], L.t.p[1] - z0, D);
    float sy = D[1], sz = D[2];
    if (D[0] != 0.0f) {
      StepJ stp;
      if (helix_step(L.r, D[0], P, stp, P.fit_max_snp)) {
        sy = sy - (stp.p0 - L.r[0]);
        sz = sz - (stp.p1 - L.r[1]);
      }
    }
    cy = L.t.p[0] - sy;
    cz = L.t.p[1] - sz;
  }
  const float wy = sqrtf(P.ext_chi2 * (L.t.c[0] + P.sy2)) * 1.001f + P.attach_margin;
  const float wz = sqrtf(P.ext_chi2 * (L.t.c[2] + P.sz2)) * 1.001f + P.attach_margin;
  if (zadd != 0.0f) cz = cz - zadd;  // the row's measured z
  const long slot = (long)f * F.nslot + js;
  int* cand = F.ft_cand + slot * kMaxCand;
  float* cchi = F.ft_cchi + slot * kMaxCand;
  int nc = 0;
  int cid[kMaxCand];
  const RowGrid g = F.rows[rr];
  for_window(F.bin_first, g, cy - wy - 0.01f, cy + wy + 0.01f, cz - wz - 0.01f, cz + wz + 0.01f,
             [&](int kk) {
    if (F.ft_fixed[kk]) return;
    const float2 pk = F.syz[kk];
    const float yk = pk.x, zk = pk.y;
    if (!(fabsf(yk - cy) <= wy && fabsf(zk - cz) <= wz)) return;
    float my, mz;
    if (!corrected(M, P, sec, L.t.x, yk, zadd != 0.0f ? zk + zadd : zk, z0, L.r, my, mz)) return;
    const float c2 = chi2_of(L.t, my, mz, P);
    if (!(c2 < P.ext_chi2)) return;
    const int id = F.sid[kk];
    int pos = nc;
    while (pos > 0 && (c2 < cchi[pos - 1] || (c2 == cchi[pos - 1] && id < cid[pos - 1]))) --pos;
    if (pos >= P.cand_k) return;
    const int lim = nc < P.cand_k ? nc : P.cand_k - 1;
    for (int j = lim; j > pos; --j) {
      cand[j] = cand[j - 1];
      cchi[j] = cchi[j - 1];
      cid[j] = cid[j - 1];
    }
    cand[pos] = kk;
    cchi[pos] = c2;
    cid[pos] = id;
    if (nc < P.cand_k) ++nc;
  });
  F.ft_ncand[slot] = (uint8_t)nc;
  F.ft_assigned[slot] = -1;
}

// Iteration 1 (inward, storing the predictions) and (kExt) the Phase III
// extrapolation below the track, as a per-lane state machine: every loop
// iteration is one station (or extrapolated row) of the lane's current track,
// and a lane whose track ends takes the next one from the work queue.  The
// next station's record is requested one step ahead.  The end state of
// iteration 1 goes to ft_end2 for k_fit2.
template <bool kMap, bool kExt>
__global__ void __launch_bounds__(256, 2) k_fit1(FrameDev F, KParams P, MapDev M, int stat) {
  if (!kMap) M.on = 0;  // (the map evaluation is compiled out)
  __shared__ float rx[kMaxRows];
  for (int r = threadIdx.x; r < P.n_rows; r += blockDim.x) rx[r] = F.row_x[r];
  __syncthreads();
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  const int nL = min(F.cnt->n_loopers, nf);
  const int NR = P.n_rows;
  int phase = kFitIdle;
  int f = 0, ns = 0, k = 0;
  bool lp = false;  // FP64 updates (low-pT looper)
  int xsec = 0;     // sector of the extrapolation
  const float4* SM = nullptr;
  float4 nxt = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float* store = nullptr;
  Lin L;
  bool done = false, all_done, first = true;
  for (;;) {
    const bool fetch = refill(phase != kFitIdle, done, all_done);
    if (all_done) break;
    if (phase == kFitIdle) {
      if (!fetch) continue;
      const int q = next_item(&F.cnt->queue[kQFit1], first, stat);
      if (q >= fit_total(nL, nf)) {
        done = true;
        continue;
      }
      const int pos = fit_position(q, nL);
      if (pos < 0) continue;
      f = F.ft_order[pos];
      lp = F.ft_looper[f] != 0;
      ns = F.ft_nst[f];
      F.ft_ok[f] = 0;
      if (ns == 0) continue;  // not reached: every chain holds clusters
      SM = F.ft_meas + (long)f * kMaxRows;
      store = F.ft_store + (long)f * kMaxRows * 5;
      nxt = SM[ns - 1];
      Trk<float> s0;
      get_state(F.st_oe + (long)F.ft_last[f] * kStateF, s0);
      lin_start(L, s0, st_sector(nxt), P);
      k = ns - 1;
      phase = kFitIn;
      continue;
    }
    if (kExt && phase == kFitExt) {
      // Phase III: one row of the inward extrapolation below the innermost
      // station (k counts the rows done; nxt: the innermost station)
      const int r = st_row(nxt) - 1 - k;
      bool go = k < P.ext_rows && r >= 0;
      if (go) go = ext_step(L, xsec, r, rx, P);
      if (go) {
        ext_candidates(F, P, M, f, kMaxInner + k, xsec * NR + r, L, F.ft_z0[f],
                       row_shift(xsec, shift_side(F, f), F.ft_zsh[f], P));
        F.ft_ext_sec[(long)f * 2 * P.ext_rows + k] = (uint16_t)xsec;
        ++k;
      } else {
        F.ft_next[f] = k;
        F.ft_ok[f] = 1;
        phase = kFitIdle;
      }
      continue;
    }
    // ---- one station
    const float4 m = nxt;
    if (k > 0) nxt = SM[k - 1];
    bool ok = true;
    if (k != ns - 1) ok = lin_goto(L, st_sector(m), rx[st_row(m)], P);
    bool have = false;
    float my = 0.0f, mz = 0.0f;
    if (ok) {
      float* st = store + k * 5;
      st[0] = L.t.p[0]; st[1] = L.t.p[1]; st[2] = L.t.c[0]; st[3] = L.t.c[1]; st[4] = L.t.c[2];
      if (st_have(m)) {
        ok = meas_at<kMap>(m, P, L.r, my, mz);
        have = ok;
      }
    }
    if (have) update_as(L.t, residual(L.t, my, mz, P), lp);
    if (!ok) {
      phase = kFitIdle;
      continue;
    }
    if (--k < 0) {
      // the end of iteration 1 starts iteration 2
      put_state(F.ft_end2 + (long)f * kStateF, L.t, L.sector);
      if (kExt) {
        k = 0;
        xsec = st_sector(nxt);
        phase = kFitExt;
      } else {
        F.ft_ok[f] = 1;
        phase = kFitIdle;
      }
    }
  }
}

// Interpolation record of inner station k of track f, from k_fit2 for k_inner_cand:
// (y, z, Cyy, Cyz, Czz, reference y, z, sin phi; the reference's tan(lambda) and
// q/pT do not change along a track, and x is the row's).  It lies where the
// station's candidates' chi2 go, which the thread that reads it then writes.
static_assert(kMaxCand * sizeof(float) == 2 * sizeof(float4), "interpolation record");
__device__ __forceinline__ float4* ipol_rec(const FrameDev& F, int f, int k) {
  return (float4*)(F.ft_cchi + ((long)f * F.nslot + k) * kMaxCand);
}

// Iteration 2 (outward) as the same kind of state machine: interpolation with
// the stored predictions, flags of outliers, inner-row candidates (Sec. 3,
// Phases I and II), then (kExt) the Phase III extrapolation above the
// outermost station.  Starts from the end of iteration 1, ends in ft_end2.  A
// flagged station's record loses its cluster (iteration 3 skips it).
enum : int { kFit2Idle = 0, kFit2St, kFit2Out };

template <bool kMap, bool kExt>
__global__ void __launch_bounds__(256, 2) k_fit2(FrameDev F, KParams P, MapDev M, int stat) {
  if (!kMap) M.on = 0;  // (the map evaluation is compiled out)
  __shared__ float rx[kMaxRows];
  for (int r = threadIdx.x; r < P.n_rows; r += blockDim.x) rx[r] = F.row_x[r];
  __syncthreads();
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  const int nL = min(F.cnt->n_loopers, nf);
  const int NR = P.n_rows;
  int phase = kFit2Idle;
  int f = 0, ns = 0, k = 0;
  bool lp = false;  // FP64 updates (low-pT looper)
  int xsec = 0;     // sector of the extrapolation
  float4* SM = nullptr;
  float4 nxt = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  const float* store = nullptr;
  float sn[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};  // the next station's prediction
  uint8_t* flag = nullptr;
  Lin L;
  bool done = false, all_done, first = true;
  for (;;) {
    const bool fetch = refill(phase != kFit2Idle, done, all_done);
    if (all_done) break;
    if (phase == kFit2Idle) {
      if (!fetch) continue;
      const int q = next_item(&F.cnt->queue[kQFit2], first, stat);
      if (q >= fit_total(nL, nf)) {
        done = true;
        continue;
      }
      const int pos = fit_position(q, nL);
      if (pos < 0) continue;
      f = F.ft_order[pos];
      if (!F.ft_ok[f]) continue;
      lp = F.ft_looper[f] != 0;
      ns = F.ft_nst[f];
      SM = F.ft_meas + (long)f * kMaxRows;
      store = F.ft_store + (long)f * kMaxRows * 5;
      flag = F.ft_flag + (long)f * kMaxRows;
      nxt = SM[0];
#pragma unroll
      for (int i = 0; i < 5; ++i) sn[i] = store[i];
      Trk<float> s1;
      get_state(F.ft_end2 + (long)f * kStateF, s1);
      lin_start(L, s1, st_sector(nxt), P);
      F.ft_ref34[f] = make_float2(L.r[3], L.r[4]);
      k = 0;
      phase = kFit2St;
      continue;
    }
    if (kExt && phase == kFit2Out) {
      // Phase III: one row of the outward extrapolation above the outermost
      // station (k counts the rows done; nxt: the outermost station)
      const int r = st_row(nxt) + 1 + k;
      bool go = k < P.ext_rows && r < NR;
      if (go) go = ext_step(L, xsec, r, rx, P);
      if (go) {
        ext_candidates(F, P, M, f, kMaxInner + P.ext_rows + k, xsec * NR + r, L, F.ft_z0[f],
                       row_shift(xsec, shift_side(F, f), F.ft_zsh[f], P));
        F.ft_ext_sec[(long)f * 2 * P.ext_rows + P.ext_rows + k] = (uint16_t)xsec;
        ++k;
      } else {
        F.ft_nout[f] = k;
        phase = kFit2Idle;
      }
      continue;
    }
    // ---- one station
    const float4 m = nxt;
    float sv[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) sv[i] = sn[i];
    if (k + 1 < ns) {
      nxt = SM[k + 1];
#pragma unroll
      for (int i = 0; i < 5; ++i) sn[i] = store[(k + 1) * 5 + i];
    }
    bool ok = true;
    if (k != 0) ok = lin_goto(L, st_sector(m), rx[st_row(m)], P);
    const bool inner = st_row(m) < P.inner_rows;
    bool have = false;
    float my = 0.0f, mz = 0.0f;
    if (ok) {
      const float a[5] = {L.t.p[0], L.t.p[1], L.t.c[0], L.t.c[1], L.t.c[2]};
      const Interp I = interpolate(a, sv);
      int fl = 0;
      if (st_have(m)) {
        ok = meas_at<kMap>(m, P, L.r, my, mz);
        have = ok;
        if (ok && !inner && chi2_interp(I, my, mz, P) > P.int_chi2) {
          fl = 1;
          SM[k].w = __uint_as_float(__float_as_uint(m.w) & ~kStHave);
        }
      }
      flag[k] = (uint8_t)fl;
      if (ok && inner) {
        // Phase II candidates of this inner station: the search runs later in
        // k_inner_cand, over all (track, inner station) pairs at once
        float4* ip = ipol_rec(F, f, k);
        ip[0] = make_float4(I.y, I.z, I.c00, I.c01);
        ip[1] = make_float4(I.c11, L.r[0], L.r[1], L.r[2]);
      }
    }
    if (have) update_as(L.t, residual(L.t, my, mz, P), lp);
    if (!ok) {
      F.ft_ok[f] = 0;
      phase = kFit2Idle;
      continue;
    }
    if (++k == ns) {
      put_state(F.ft_end2 + (long)f * kStateF, L.t, L.sector);
      k = 0;
      xsec = st_sector(nxt);
      phase = kExt ? kFit2Out : kFit2Idle;
    }
  }
}

// Second ambiguity solving, round k: bids (chi2, track key) per free cluster.
__device__ __forceinline__ bool inner_station(const FrameDev& F, const KParams& P, int f, int k) {
  return k < F.ft_nst[f] && (F.ft_st_rs[(long)f * kMaxRows + k] % P.n_rows) < P.inner_rows;
}

// Phase II candidate search of every inner station of every fit track, from
// the interpolation k_fit2 left for it (one thread per (track, station)).
template <bool kMap>
__global__ void k_inner_cand(FrameDev F, KParams P, MapDev M) {
  if (!kMap) M.on = 0;  // (the map evaluation is compiled out: 48 registers instead of 110)
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  const long tot = (long)nf * P.inner_rows;
  for (long w = (long)blockIdx.x * blockDim.x + threadIdx.x; w < tot;
       w += (long)gridDim.x * blockDim.x) {
    const int f = (int)(w / P.inner_rows), k = (int)(w % P.inner_rows);
    if (!F.ft_ok[f] || !inner_station(F, P, f, k)) {
      F.ft_ncand[(long)f * F.nslot + k] = 0;  // (the ambiguity looks at the count only)
      continue;
    }
    const float4* ip = ipol_rec(F, f, k);
    const float4 u = ip[0], v = ip[1];
    const float2 w34 = F.ft_ref34[f];
    const Interp I{u.x, u.y, u.z, u.w, v.x};
    const float ref[5] = {v.y, v.z, v.w, w34.x, w34.y};
    const int rs = F.ft_st_rs[(long)f * kMaxRows + k];
    inner_candidates(F, P, M, f, k, rs, F.row_x[rs % P.n_rows], ref, I, F.ft_z0[f],
                     row_shift(rs / P.n_rows, shift_side(F, f), F.ft_zsh[f], P));
  }
}

// Work item w of the second ambiguity: (fit track, candidate slot).  Slots
// 0..inner_rows-1 are the inner stations, the next ext_rows slots the rows
// extrapolated below the track, the ext_rows after them the rows extrapolated
// above it (Phase III); returns -1 for an unused extrapolation slot (an unused
// inner slot has no candidates).
__device__ __forceinline__ int amb_per(const KParams& P) { return P.inner_rows + 2 * P.ext_rows; }

__device__ __forceinline__ long amb_slot(const FrameDev& F, const KParams& P, long w, int& f,
                                         int& k) {
  const int per = amb_per(P);
  f = (int)(w / per);
  k = (int)(w % per);
  if (k < P.inner_rows) return (long)f * F.nslot + k;
  if (!F.ft_ok[f]) return -1;
  const int e = k - P.inner_rows;
  if (e < P.ext_rows) return e < F.ft_next[f] ? (long)f * F.nslot + kMaxInner + e : -1;
  const int eo = e - P.ext_rows;
  return eo < F.ft_nout[f] ? (long)f * F.nslot + kMaxInner + P.ext_rows + eo : -1;
}

__global__ void k_amb_bid(FrameDev F, KParams P, int round) {
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  const long tot = (long)nf * amb_per(P);
  for (long w = (long)blockIdx.x * blockDim.x + threadIdx.x; w < tot;
       w += (long)gridDim.x * blockDim.x) {
    int f, k;
    const long sk = amb_slot(F, P, w, f, k);
    if (sk < 0 || F.ft_ncand[sk] <= round || F.ft_assigned[sk] >= 0) continue;
    const int c = F.ft_cand[sk * kMaxCand + round];
    if (F.taken[c]) continue;
    atomicMin(&F.bid[c], pack_chi_key(F.ft_cchi[sk * kMaxCand + round], F.ft_key[f]));
  }
}

// The round's winners: the slot whose own (chi2, track key) is the cluster's
// lowest bid takes it, marks it taken and empties the bid again.  Keys are
// unique per track and a track lists a cluster once, so every bid has one winner,
// and a slot that reads the bid or the mark after its winner changed them loses,
// as it would before.  The last round (kLast) also brings the inner stations'
// measurements in line with the clusters they were given, for iteration 3.
template <bool kLast, bool kMap>
__global__ void k_amb_resolve(FrameDev F, KParams P, MapDev M, int round) {
  if (!kMap) M.on = 0;
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  const long tot = (long)nf * amb_per(P);
  for (long w = (long)blockIdx.x * blockDim.x + threadIdx.x; w < tot;
       w += (long)gridDim.x * blockDim.x) {
    int f, k;
    const long sk = amb_slot(F, P, w, f, k);
    if (sk < 0) continue;
    const bool more = F.ft_ncand[sk] > round;
    if (!kLast && !more) continue;
    // (an unused inner slot: ncand is 0, assigned and ft_ok stand for themselves)
    int got = F.ft_assigned[sk];
    if (more && got < 0) {
      const int c = F.ft_cand[sk * kMaxCand + round];
      if (!F.taken[c] &&
          F.bid[c] == pack_chi_key(F.ft_cchi[sk * kMaxCand + round], F.ft_key[f])) {
        F.ft_assigned[sk] = got = c;
        F.taken[c] = 1;
        F.bid[c] = ~0ull;
      }
    }
    if (kLast && k < P.inner_rows && F.ft_ok[f] && inner_station(F, P, f, k)) {
      float4* m = F.ft_meas + (long)f * kMaxRows + k;
      if (got < 0) {
        m->w = __uint_as_float(__float_as_uint(m->w) & ~kStHave);
      } else if (got != F.ft_st_cl[(long)f * kMaxRows + k]) {
        const int rs = F.ft_st_rs[(long)f * kMaxRows + k];
        const float2 pc = F.syz[got];
        *m = fit_meas<kMap>(M, P, rs, F.row_x[rs % P.n_rows], pc.x,
                            track_z(pc.y, rs / P.n_rows, shift_side(F, f), F.ft_zsh[f], P),
                            F.ft_z0[f]);
      }
    }
  }
}

// Iteration 3: inward with the surviving and re-attached clusters (as the
// station records hold them after iteration 2 and the second ambiguity
// solving), simple cut.
template <bool kMap, bool kExt>
__global__ void __launch_bounds__(256, 2) k_fit3(FrameDev F, KParams P, MapDev M, int stat) {
  if (!kMap) M.on = 0;  // (the map evaluation is compiled out)
  __shared__ float rx[kMaxRows];
  for (int r = threadIdx.x; r < P.n_rows; r += blockDim.x) rx[r] = F.row_x[r];
  __syncthreads();
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  const int NR = P.n_rows;
  const int nL = min(F.cnt->n_loopers, nf);
  bool first = true;
  for (;;) {
    const int q = next_item(&F.cnt->queue[kQFit3], first, stat);
    if (q >= fit_total(nL, nf)) break;
    const int pos = fit_position(q, nL);
    if (pos < 0) continue;
    const int f = F.ft_order[pos];
    const bool lp = F.ft_looper[f] != 0;  // FP64 updates (low-pT looper)
    F.ft_n[f] = 0;
    if (!F.ft_ok[f]) continue;
    const int ns = F.ft_nst[f];
    const int* SC = F.ft_st_cl + (long)f * kMaxRows;
    const float4* SM = F.ft_meas + (long)f * kMaxRows;
    int* used = F.ft_used + (long)f * kMaxRows;
    const float z0 = F.ft_z0[f];
    const float zsh = F.ft_zsh[f];
    const int zside = shift_side(F, f);
    Trk<float> s2;
    const float* e2 = F.ft_end2 + (long)f * kStateF;
    get_state(e2, s2);
    float4 nxt = SM[ns - 1];
    Lin L;
    lin_start(L, s2, st_sector(nxt), P);
    float chi2 = 0.0f;
    int n = 0;
    Trk<float> out = L.t;
    int out_sec = L.sector;
    bool have = false;
    // Phase III outward rows: each assigned cluster is tested and filtered
    // against a forward extrapolation of the iteration-2 end state (its own
    // covariance), so that it joins the track without moving the fit of the
    // stations; in the list the outward clusters precede the stations
    const int nout = kExt ? F.ft_nout[f] : 0;
    if (kExt && nout > 0) {
      const int secl = st_sector(nxt), rl = st_row(nxt);
      Lin E;
      E.t = s2;
#pragma unroll
      for (int i = 0; i < 5; ++i) E.r[i] = s2.p[i];
      E.sector = secl;
      const long o0 = (long)f * F.nslot + kMaxInner + P.ext_rows;
      const uint16_t* xs = F.ft_ext_sec + (long)f * 2 * P.ext_rows + P.ext_rows;
      for (int e = 0; e < nout; ++e) {
        const int sx = xs[e];
        if (!lin_goto(E, sx, rx[rl + 1 + e], P)) break;
        const int c = F.ft_assigned[o0 + e];
        if (c < 0) continue;
        const float2 pc = F.syz[c];
        float my, mz;
        if (!corrected(M, P, sx, E.t.x, pc.x, track_z(pc.y, sx, zside, zsh, P), z0, E.r, my,
                       mz))
          continue;
        const Resid R = residual(E.t, my, mz, P);
        if (R.chi2 > P.final_chi2) continue;
        chi2 = chi2 + R.chi2;
        update_as(E.t, R, lp);
        used[n] = c;
        ++n;
      }
      for (int i = 0, j = n - 1; i < j; ++i, --j) {  // outermost first
        const int u = used[i];
        used[i] = used[j];
        used[j] = u;
      }
    }
    // the stations inward, then the rows extrapolated below the innermost one
    const int next = kExt ? F.ft_next[f] : 0;
    for (int k = ns - 1; k >= -next; --k) {
      // the station's record is requested one step ahead, its cluster's index
      // before the station change; inner stations hold at most inner_rows <=
      // kMaxInner entries, as rows increase along a track
      int sec, row, c;
      float4 m = nxt;
      if (!kExt || k >= 0) {
        if (k > 0) nxt = SM[k - 1];
        sec = st_sector(m);
        row = st_row(m);
        c = -1;
        if (st_have(m)) c = row < P.inner_rows ? F.ft_assigned[(long)f * F.nslot + k] : SC[k];
      } else {  // nxt: the innermost station
        sec = F.ft_ext_sec[(long)f * 2 * P.ext_rows - 1 - k];
        row = st_row(nxt) + k;
        c = F.ft_assigned[(long)f * F.nslot + kMaxInner - 1 - k];
        if (c >= 0) {
          const float2 pc = F.syz[c];
          m = fit_meas<kMap>(M, P, sec * NR + row, rx[row], pc.x,
                             track_z(pc.y, sec, zside, zsh, P), z0);
        } else {
          m.w = 0.0f;
        }
      }
      if (k != ns - 1 && !lin_goto(L, sec, rx[row], P)) break;
      if (!st_have(m)) continue;
      float my, mz;
      if (!meas_at<kMap>(m, P, L.r, my, mz)) continue;
      const Resid R = residual(L.t, my, mz, P);
      if (R.chi2 > P.final_chi2) continue;
      chi2 = chi2 + R.chi2;
      update_as(L.t, R, lp);
      used[n] = c;
      ++n;
      out = L.t;
      out_sec = L.sector;
      have = true;
    }
    F.ft_n[f] = have ? n : 0;
    F.ft_chi2[f] = chi2;
    put_state(F.ft_out + (long)f * kStateF, out, out_sec);
  }
}

// ------------------------------------------------------------ a11 outputs
__device__ __forceinline__ int out_flag(const FrameDev& F, const KParams& P, int f, int nf) {
  return (f < nf && F.ft_ok[f] && F.ft_n[f] >= P.min_hits) ? 1 : 0;
}

__global__ void k_out_count(FrameDev F, KParams P) {
  __shared__ int sh[32];
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  const int fl = F.cnt->err ? 0 : out_flag(F, P, f, nf);
  const int v = fl ? F.ft_n[f] : 0;
  int tot_t, tot_r;
  block_exscan(fl, sh, &tot_t);
  block_exscan(v, sh, &tot_r);
  if (threadIdx.x == 0) {
    F.scan_tmp[2 * blockIdx.x] = tot_t;
    F.scan_tmp[2 * blockIdx.x + 1] = tot_r;
  }
}

// Exclusive scan of the interleaved (tracks, refs) block partials.
__global__ void k_out_scan(FrameDev F, int nparts) {
  __shared__ int sh[32];
  __shared__ int ct, cr;
  if (threadIdx.x == 0) { ct = 0; cr = 0; }
  __syncthreads();
  for (int base = 0; base < nparts; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const int vt = i < nparts ? F.scan_tmp[2 * i] : 0;
    const int vr = i < nparts ? F.scan_tmp[2 * i + 1] : 0;
    int tt, tr;
    const int et = block_exscan(vt, sh, &tt);
    const int er = block_exscan(vr, sh, &tr);
    if (i < nparts) {
      F.scan_tmp[2 * i] = ct + et;
      F.scan_tmp[2 * i + 1] = cr + er;
    }
    __syncthreads();
    if (threadIdx.x == 0) { ct += tt; cr += tr; }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    F.cnt->n_refs = cr;
    F.cnt->n_out = ct;
  }
}

__global__ void k_out_write(FrameDev F, KParams P) {
  __shared__ int sh[32];
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  const int fl = F.cnt->err ? 0 : out_flag(F, P, f, nf);
  const int v = fl ? F.ft_n[f] : 0;
  int tt, tr;
  const int et = block_exscan(fl, sh, &tt);
  const int er = block_exscan(v, sh, &tr);
  if (!fl) {
    if (f < nf) F.ft_outidx[f] = -1;
  } else {
    const int t = F.scan_tmp[2 * blockIdx.x] + et;
    const int off = F.scan_tmp[2 * blockIdx.x + 1] + er;
    F.ft_outidx[f] = t;
    const float* o = F.ft_out + (long)f * kStateF;
    for (int i = 0; i < 5; ++i) F.out_par[(long)t * 5 + i] = o[i];
    for (int i = 0; i < 15; ++i) F.out_cov[(long)t * 15 + i] = o[5 + i];
    F.out_x[t] = o[20];
    F.out_zsh[t] = F.ft_zsh[f];
    F.out_sector[t] = __float_as_int(o[21]);
    F.out_chi2[t] = F.ft_chi2[f];
    F.out_ndf[t] = 2 * v - 5;
    F.out_ncl[t] = v;
    F.out_key[t] = F.ft_key[f];
    F.out_offset[t] = off;
    if ((long)off + v > F.cap_refs) atomicOr(&F.cnt->err, kErrCapRefs);
  }
}

// Cluster lists: a warp takes its lanes' tracks one by one, its lanes over the
// track's clusters (the used list read innermost first, all loads issued before
// the ids they address), writing the input ids 32 at a time and lowering their
// attachment keys.
__global__ void k_out_lists(FrameDev F) {
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  constexpr int kChunks = (kMaxRows + 31) / 32;
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (blockDim.x >> 5);
  const int per = warp_share(nf, nw);
  for (int f0 = per * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); f0 < nf;
       f0 += per * nw) {
    const int f = f0 + lane;
    int t = -1, v = 0, off = 0, key = 0;
    if (lane < per && f < nf) t = F.ft_outidx[f];
    if (t >= 0) {
      v = F.ft_n[f];
      key = F.ft_key[f];
      off = F.out_offset[t];
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, t >= 0); todo; todo &= todo - 1) {
      const int j = __ffs(todo) - 1;
      const int nj = __shfl_sync(0xffffffffu, v, j);
      const int oj = __shfl_sync(0xffffffffu, off, j);
      const int kj = __shfl_sync(0xffffffffu, key, j);
      const bool fits = (long)oj + nj <= F.cap_refs;
      const int* used = F.ft_used + (long)(f0 + j) * kMaxRows;
      int u[kChunks], id[kChunks];
#pragma unroll
      for (int c = 0; c < kChunks; ++c) {
        const int q = lane + 32 * c;
        u[c] = q < nj ? used[nj - 1 - q] : -1;
      }
#pragma unroll
      for (int c = 0; c < kChunks; ++c) id[c] = u[c] >= 0 ? F.sid[u[c]] : -1;
#pragma unroll
      for (int c = 0; c < kChunks; ++c) {
        if (id[c] < 0) continue;
        if (fits) F.out_ids[oj + lane + 32 * c] = id[c];
        atomicMin(&F.attach_key[id[c]], kj);
      }
    }
  }
}

// Attachment: every cluster goes to the track with the smallest key among
// those that use it.  A warp takes up to 32 consecutive fit tracks one by one,
// the lanes over the track's clusters.
__global__ void k_out_attach(FrameDev F, KParams P) {
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  if (F.cnt->err) return;
  constexpr int kChunks = (kMaxRows + 31) / 32;
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (blockDim.x >> 5);
  const int per = warp_share(nf, nw);
  for (int f0 = per * (blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)); f0 < nf;
       f0 += per * nw) {
    const int f = f0 + lane;
    int t = -1, n = 0, key = 0, off = 0;
    if (lane < per && f < nf) {
      t = F.ft_outidx[f];
      if (t >= 0) {
        n = F.ft_n[f];
        key = F.ft_key[f];
        off = F.out_offset[t];
        if (t == F.cnt->n_out - 1) F.out_offset[t + 1] = F.cnt->n_refs;
      }
    }
    for (unsigned todo = __ballot_sync(0xffffffffu, t >= 0); todo; todo &= todo - 1) {
      const int j = __ffs(todo) - 1;
      const int tj = __shfl_sync(0xffffffffu, t, j);
      const int nj = __shfl_sync(0xffffffffu, n, j);
      const int kj = __shfl_sync(0xffffffffu, key, j);
      const int oj = __shfl_sync(0xffffffffu, off, j);
      const int* ids = F.out_ids + oj;
      int id[kChunks], ak[kChunks];
#pragma unroll
      for (int c = 0; c < kChunks; ++c) {
        const int q = lane + 32 * c;
        id[c] = q < nj ? ids[q] : -1;
      }
#pragma unroll
      for (int c = 0; c < kChunks; ++c) ak[c] = id[c] >= 0 ? F.attach_key[id[c]] : 0;
#pragma unroll
      for (int c = 0; c < kChunks; ++c)
        if (id[c] >= 0 && ak[c] == kj) F.attach[id[c]] = tj;
    }
  }
}

// ------------------------------------------- a12 refit with fixed clusters
// Tracks merged across the central electrode carry the shift of their far
// side (in_zsh): zsh and the side whose clusters take it (zside, -1: none;
// the other side than the innermost cluster's), for track_z.
__device__ __forceinline__ void refit_shift(const RefitDev& R, const KParams& P, int t,
                                            float& zsh, int& zside) {
  zsh = R.in_zsh ? R.in_zsh[t] : 0.0f;
  zside = zsh != 0.0f ? 1 - ((R.sector[R.ids[R.offset[t]]] / P.n_phi) & 1) : -1;
}
__device__ __forceinline__ void save_ckpt(float* d, const Lin& L) {
#pragma unroll
  for (int i = 0; i < 5; ++i) d[i] = L.t.p[i];
#pragma unroll
  for (int i = 0; i < 15; ++i) d[5 + i] = L.t.c[i];
#pragma unroll
  for (int i = 0; i < 5; ++i) d[20 + i] = L.r[i];
  d[25] = L.t.x;
  d[26] = __int_as_float(L.sector);
}

__device__ __forceinline__ void load_ckpt(const float* d, Lin& L) {
#pragma unroll
  for (int i = 0; i < 5; ++i) L.t.p[i] = d[i];
#pragma unroll
  for (int i = 0; i < 15; ++i) L.t.c[i] = d[5 + i];
#pragma unroll
  for (int i = 0; i < 5; ++i) L.r[i] = d[20 + i];
  L.t.x = d[25];
  L.sector = __float_as_int(d[26]);
}

__device__ __forceinline__ void lin_start2(Lin& L, const Trk<float>& s, const float* ref,
                                           int sector, const KParams& P) {
  L.t = s;
  reset_cov(L.t.c, P);
#pragma unroll
  for (int i = 0; i < 5; ++i) L.r[i] = ref[i];
  L.sector = sector;
}

// Forward refit (see the oracle's definition): extended-Kalman start pass on
// uncorrected clusters, then iterations 1-3 with checkpoints of the filter
// (state, covariance, reference) every kCkptStride stations.  First, one warp
// per track, the lanes over its clusters: each reference's position in the
// frame of the track's innermost side and its correction, which depend on no
// filter state and would otherwise be evaluated in every pass on the serial
// chain of the track's steps.  Then four kernels, one per pass, each a
// per-lane state machine (a step per loop iteration, refilled from a work
// queue), each leaving the next one's start in that pass's first checkpoint.
// (As one kernel of four loops per track the lanes of a warp did not reconverge:
// 4.9 ms for the 3,900 tracks of an event in strict mode.)
// R.ok counts the passes done: a pass takes a track only if the one before it
// succeeded (-1 from the preparation: a cluster's row is none of the detector's,
// and the passes hold the rows' x in shared memory; the track is not fitted).
__global__ void __launch_bounds__(256, 2) k_refit_prep(RefitDev R, KParams P, int* steps3) {
  const MapDev M = R.map;
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (blockDim.x >> 5);
  for (int t = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < R.n_tracks; t += nw) {
    const int o0 = R.offset[t], ns = R.offset[t + 1] - o0;
    const float* ip = R.in_par + (long)t * 5;
    const float inx = R.in_x[t];
    const float z0 = ip[1] - ip[3] * sqrtf(inx * inx + ip[0] * ip[0]);
    if (lane == 0) {
      R.ok[t] = 0;
      R.nused[t] = 0;
      R.chi2[t] = 0.0f;
      steps3[t] = 0;
      R.z0[t] = z0;
    }
    if (ns < 1 || ns > kMaxRows) continue;
    float zsh;
    int zside;
    refit_shift(R, P, t, zsh, zside);
    bool bad = false;
    for (int k = lane; k < ns; k += 32) {
      const int c = R.ids[o0 + k];
      const int s = R.sector[c], row = R.row[c];
      const float y = R.y[c], z = track_z(R.z[c], s, zside, zsh, P);
      float4 m = make_float4(0.0f, y, z, __int_as_float(s << 8 | row));
      if (row >= P.n_rows) {
        bad = true;
      } else if (M.on) {
        float D[3];
        map_eval<true>(M, P, s, R.row_x[row], y, z - z0, D);
        m.x = D[0];
        m.y = y + D[1];
        m.z = z + D[2];
      }
      R.raw[o0 + k] = make_float2(y, z);
      R.meas[o0 + k] = m;
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) R.ok[t] = -1;
  }
}

// Order of the tracks for the four passes, stretch by stretch: loopers (by
// their start parameters; the passes judge at every update) first, each part by
// clusters, so that the lanes of a warp run the same update and end together.
__global__ void __launch_bounds__(kBlock) k_refit_order(RefitDev R, KParams P) {
  constexpr int kHalf = kOrdBuckets / 2;
  for (int c0 = blockIdx.x * kOrdChunk; c0 < R.n_tracks; c0 += gridDim.x * kOrdChunk)
    order_chunk(
        (int)min((long)kOrdChunk, R.n_tracks - c0), [&](int q) { return c0 + q; },
        [&](int t) {
          const int ns = max(0, min(kMaxRows, R.offset[t + 1] - R.offset[t]));
          const bool looper =
              P.looper_qpt > 0.0f && fabsf(R.in_par[(long)t * 5 + 4]) > P.looper_qpt;
          return (looper ? kHalf - 1 : -1) + min(kHalf - 1, ns * kHalf / kMaxRows);
        },
        R.order + c0);
}

__device__ __forceinline__ float* refit_ckpt(const RefitDev& R, int t, int it, int seg) {
  return R.ckpt + (((long)t * 3 + it) * kCkptSeg + seg) * kCkptF;
}

__global__ void __launch_bounds__(128, 4) k_refit_start(RefitDev R, KParams P, int stat) {
  __shared__ float rx[kMaxRows];
  for (int r = threadIdx.x; r < P.n_rows; r += blockDim.x) rx[r] = R.row_x[r];
  __syncthreads();
  const int half = P.n_phi;
  bool busy = false, first = true;
  int t = 0, k = 0, ns = 0, sec = 0;
  const float2* raw = nullptr;
  const float4* meas = nullptr;
  float2 nyz = make_float2(0.0f, 0.0f);
  int nw = 0;
  Trk<float> t0;
  for (;;) {
    if (!busy) {
      t = next_item(&R.queue[0], first, stat);
      if (t >= R.n_tracks) break;
      t = R.order[t];
      const int o0 = R.offset[t];
      ns = R.offset[t + 1] - o0;
      if (ns < 1 || ns > kMaxRows) continue;
      if (R.ok[t] < 0) {
        R.ok[t] = 0;
        continue;
      }
      raw = R.raw + o0;
      meas = R.meas + o0;
      nyz = raw[0];
      nw = __float_as_int(meas[0].w);
#pragma unroll
      for (int i = 0; i < 5; ++i) t0.p[i] = R.in_par[(long)t * 5 + i];
      t0.x = R.in_x[t];
      reset_cov(t0.c, P);
      sec = R.in_sector[t];
      k = 0;
      busy = true;
      continue;
    }
    const float2 yz = nyz;
    const int s = nw >> 8, row = nw & 0xFF;
    if (k + 1 < ns) {
      nyz = raw[k + 1];
      nw = __float_as_int(meas[k + 1].w);
    }
    bool ok = true;
    if (s != sec) {
      const int ds = ((s % half) - (sec % half) + half) % half;
      // ds == 0: the same azimuthal sector across the central electrode
      if ((ds != 0 && ds != 1 && ds != half - 1) ||
          (ds != 0 && !rotate(t0, ds == 1 ? 1 : -1, P, P.fit_max_snp)))
        ok = false;
      sec = s;
    }
    if (ok) ok = propagate(t0, rx[row], P, P.fit_max_snp);
    if (!ok) {
      busy = false;
      continue;
    }
    update(t0, residual(t0, yz.x, yz.y, P));
    if (++k < ns) continue;
    Lin L;
    lin_start(L, t0, s, P);
    save_ckpt(refit_ckpt(R, t, 0, 0), L);
    R.ok[t] = 1;
    busy = false;
  }
}

// Iteration IT of the refit (0: inward, 1: outward with the interpolation
// flags, 2: inward with the cuts).
template <int IT, bool kMap>
__global__ void __launch_bounds__(128, 4) k_refit_iter(RefitDev R, KParams P, int* steps3, int stat) {
  __shared__ float rx[kMaxRows];
  for (int r = threadIdx.x; r < P.n_rows; r += blockDim.x) rx[r] = R.row_x[r];
  __syncthreads();
  bool busy = false, first = true;
  int t = 0, j = 0, ns = 0, o0 = 0, n = 0, out_sec = 0;
  const float4* meas = nullptr;
  float4 nxt = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  float* store = nullptr;
  float sn[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};  // the next station's prediction
  float chi2 = 0.0f;
  Lin L;
  Trk<float> out;  // the state after the last cluster used
  for (;;) {
    if (!busy) {
      t = next_item(&R.queue[1 + IT], first, stat);
      if (t >= R.n_tracks) break;
      t = R.order[t];
      if (R.ok[t] != IT + 1) continue;
      o0 = R.offset[t];
      ns = R.offset[t + 1] - o0;
      meas = R.meas + o0;
      store = R.store + (long)t * kMaxRows * 5;
      nxt = meas[IT == 1 ? 0 : ns - 1];
      if (IT == 1) {
#pragma unroll
        for (int i = 0; i < 5; ++i) sn[i] = store[i];
      }
      load_ckpt(refit_ckpt(R, t, IT, 0), L);
      if (IT == 2) {
        chi2 = 0.0f;
        n = 0;
        out = L.t;
        out_sec = L.sector;
      }
      j = 0;
      busy = true;
      continue;
    }
    const int k = IT == 1 ? j : ns - 1 - j;
    const float4 m = nxt;
    const int w = __float_as_int(m.w);
    float sv[5];
    if (IT == 1) {
#pragma unroll
      for (int i = 0; i < 5; ++i) sv[i] = sn[i];
    }
    bool skip = false, keep = false;
    if (IT == 2) {
      skip = R.flag[o0 + k] != 0;
      if (R.freeze) keep = R.acc[o0 + k] != 0;
    }
    if (j + 1 < ns) {
      nxt = meas[IT == 1 ? k + 1 : k - 1];
      if (IT == 1) {
#pragma unroll
        for (int i = 0; i < 5; ++i) sn[i] = store[(k + 1) * 5 + i];
      }
    }
    if (j > 0 && j % kCkptStride == 0) save_ckpt(refit_ckpt(R, t, IT, j / kCkptStride), L);
    bool ok = true;
    if (j != 0) ok = lin_goto(L, w >> 8, rx[w & 0xFF], P);
    float my = 0.0f, mz = 0.0f;
    Interp I;
    if (IT < 2) {
      if (ok) {
        if (IT == 0) {
          float* st = store + k * 5;
          st[0] = L.t.p[0]; st[1] = L.t.p[1]; st[2] = L.t.c[0]; st[3] = L.t.c[1];
          st[4] = L.t.c[2];
        }
        if (IT == 1) {
          const float a[5] = {L.t.p[0], L.t.p[1], L.t.c[0], L.t.c[1], L.t.c[2]};
          I = interpolate(a, sv);
        }
        ok = meas_at<kMap>(m, P, L.r, my, mz);
      }
      if (!ok) {
        R.ok[t] = 0;
        busy = false;
        continue;
      }
      if (IT == 1 && !R.freeze) {
        R.flag[o0 + k] = chi2_interp(I, my, mz, P) > P.int_chi2 ? 1 : 0;
      }
      fit_update(L.t, residual(L.t, my, mz, P), P);
      if (++j < ns) continue;
      // the end of this pass starts the next, about the reference kept for it
      float* ref = R.ref + (long)t * 10 + 5 * IT;
      if (!R.freeze) {
#pragma unroll
        for (int i = 0; i < 5; ++i) ref[i] = L.t.p[i];
      }
      const Trk<float> s = L.t;
      lin_start2(L, s, ref, w >> 8, P);
      save_ckpt(refit_ckpt(R, t, IT + 1, 0), L);
      R.ok[t] = IT + 2;
      busy = false;
      continue;
    }
    if (ok && !skip && meas_at<kMap>(m, P, L.r, my, mz)) {
      const Resid Rs = residual(L.t, my, mz, P);
      const bool accept = R.freeze ? keep : !(Rs.chi2 > P.final_chi2);
      if (!R.freeze) R.acc[o0 + k] = accept ? 1 : 0;
      if (accept) {
        chi2 = chi2 + Rs.chi2;
        fit_update(L.t, Rs, P);
        ++n;
        out = L.t;
        out_sec = L.sector;
      }
    }
    if (ok && ++j < ns) continue;
    steps3[t] = j;
    R.ok[t] = n > 0 ? 1 : 0;
    R.nused[t] = n;
    R.chi2[t] = chi2;
    R.ndf[t] = 2 * n - 5;
    R.out_sector[t] = out_sec;
    R.out_x[t] = out.x;
#pragma unroll
    for (int i = 0; i < 5; ++i) R.out_par[(long)t * 5 + i] = out.p[i];
#pragma unroll
    for (int i = 0; i < 15; ++i) R.out_cov[(long)t * 15 + i] = out.c[i];
    busy = false;
  }
}

// Adjoint of the refit: d(sum_t w_t chi2_t)/d(map) with references and
// decisions held fixed, in three kernels per chunk of tracks:
//  k_refit_replay   one thread per (track, iteration, segment of kCkptStride
//                   stations): the segment's filter steps recomputed from its
//                   checkpoint, with identical arithmetic, each leaving what
//                   the reverse sweep needs of it in a 96-byte record.  The
//                   segments do not depend on one another, so 30 times as many
//                   threads as tracks share this (most of the arithmetic);
//  k_refit_reverse  one thread per track over iterations 3, 2, 1 in reverse:
//                   five adjoint words and some thirty operations per step,
//                   leaving the gradient by the step's corrected cluster;
//  k_refit_scatter  those gradients through the 64 spline weights into FP64
//                   accumulators (the cross-track reduction in FP64), summed
//                   over the blocks in a fixed order by k_grad_reduce.
// (As one kernel with a thread per track, the steps of a segment in local
// memory and 192 FP64 shared-memory atomics per cluster, its 138 KB of
// accumulators left 8 warps per SM: 17 ms for the 7,500 tracks of a distorted
// 1.2e6-cluster frame.)
//
// Step record: F (f02, f04, f12, f13, f14, f24), W r of a step counted in
// chi2 (else 0), d(measurement)/d(x displacement), gain columns k0 and k1, the
// rotation's (j00, j10, j20, j22) (else the identity's); zeros where a step has
// no propagation or no update.  The reverse sweep replaces the first float4 by
// the gradient by the step's (x displacement, y, z).
__device__ __forceinline__ float4* adj_rec(const RefitDev& R, int q) {  // track q of the chunk
  return R.rec + (long)q * 3 * kMaxRows * kRecV;
}

__global__ void __launch_bounds__(128, 4) k_refit_replay(RefitDev R, KParams P,
                                                         const int* steps3, int t0, int tn) {
  const long wk = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (wk >= (long)tn * 3 * kCkptSeg) return;
  // (a warp's lanes: 32 neighbouring tracks in one segment and iteration)
  const int t = t0 + (int)(wk % tn);
  const int it = (int)(wk / tn) % 3, sg = (int)(wk / tn) / 3;
  if (!R.ok[t]) return;
  const int o0 = R.offset[t], ns = R.offset[t + 1] - o0;
  const int nsteps = it == 2 ? steps3[t] : ns;
  const int j0 = sg * kCkptStride, j1 = min(nsteps, j0 + kCkptStride);
  if (j0 >= nsteps) return;
  float4* rec = adj_rec(R, t - t0) + (long)it * ns * kRecV;
  Lin L;
  load_ckpt(refit_ckpt(R, t, it, sg), L);
  for (int j = j0; j < j1; ++j) {
    const int k = it == 1 ? j : ns - 1 - j;
    const float4 m = R.meas[o0 + k];
    const int w = __float_as_int(m.w);
    StepJ S;
    S.f02 = S.f04 = S.f12 = S.f13 = S.f14 = S.f24 = 0.0f;
    float jr[4] = {1.0f, 0.0f, 0.0f, 1.0f};
    float k0[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f}, k1[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    float q0 = 0.0f, q1 = 0.0f, gy = 0.0f, gz = 0.0f;
    bool go = true;
    if (j != 0) go = lin_goto(L, w >> 8, R.row_x[w & 0xFF], P, jr, &S);
    if (go && !(it == 2 && (R.flag[o0 + k] || !R.acc[o0 + k]))) {
      // the measurement with its derivative by the x displacement
      float my = m.y, mz = m.z, snp1 = L.r[2];
      if (m.x != 0.0f) {
        StepJ st;
        go = helix_step(L.r, m.x, P, st, P.fit_max_snp);
        if (go) {
          my = my - (st.p0 - L.r[0]);
          mz = mz - (st.p1 - L.r[1]);
          snp1 = st.p2;
        }
      }
      if (go) {  // (iteration 3 skips a cluster that the reference cannot reach)
        const float csp1 = sqrtf(1.0f - snp1 * snp1);
        gy = -snp1 / csp1;
        gz = -L.r[3] / csp1;
        const Resid Rs = residual(L.t, my, mz, P);
        const float h0[5] = {L.t.c[0], L.t.c[1], L.t.c[3], L.t.c[6], L.t.c[10]};
        const float h1[5] = {L.t.c[1], L.t.c[2], L.t.c[4], L.t.c[7], L.t.c[11]};
#pragma unroll
        for (int i = 0; i < 5; ++i) {
          k0[i] = h0[i] * Rs.w00 + h1[i] * Rs.w01;
          k1[i] = h0[i] * Rs.w01 + h1[i] * Rs.w11;
        }
        if (it == 2) {
          q0 = Rs.w00 * Rs.r0 + Rs.w01 * Rs.r1;
          q1 = Rs.w01 * Rs.r0 + Rs.w11 * Rs.r1;
        }
        fit_update(L.t, Rs, P);
      }
    }
    float4* r = rec + (long)j * kRecV;
    r[0] = make_float4(S.f02, S.f04, S.f12, S.f13);
    r[1] = make_float4(S.f14, S.f24, q0, q1);
    r[2] = make_float4(gy, gz, k0[0], k0[1]);
    r[3] = make_float4(k0[2], k0[3], k0[4], k1[0]);
    r[4] = make_float4(k1[1], k1[2], k1[3], k1[4]);
    r[5] = make_float4(jr[0], jr[1], jr[2], jr[3]);
  }
}

// The records of kRevStage steps are copied to shared memory one stage ahead
// (16-byte asynchronous copies, each thread its own track's records, laid out
// so that a warp's reads hit distinct banks): the sweep is a serial chain of
// steps, and each step's loads would otherwise stand in it.
constexpr int kRevStage = 8;
constexpr int kRevBlock = 64;

__device__ __forceinline__ void copy_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (unsigned)__cvta_generic_to_shared(smem)),
               "l"(gmem)
               : "memory");
}

__global__ void __launch_bounds__(kRevBlock) k_refit_reverse(RefitDev R, const int* steps3, int t0,
                                                             int tn) {
  extern __shared__ float4 rev_sh[];  // [2][kRevStage * kRecV][kRevBlock]
  const int q = blockIdx.x * kRevBlock + threadIdx.x;
  if (q >= tn || !R.ok[t0 + q]) return;
  const int t = t0 + q;
  const int ns = R.offset[t + 1] - R.offset[t];
  const int tot = 2 * ns + steps3[t];
  const float w2 = 2.0f * R.dl_dchi2[t];
  float4* rec = adj_rec(R, q);
  float4* const sh = rev_sh + threadIdx.x;
  auto fetch = [&](int s) {  // stage s: steps tot - 1 - s kRevStage downwards
    float4* d = sh + (s & 1) * (kRevStage * kRecV * kRevBlock);
    for (int e = 0; e < kRevStage; ++e) {
      const int i = tot - 1 - s * kRevStage - e;
      if (i < 0) break;
#pragma unroll
      for (int v = 0; v < kRecV; ++v)
        copy_async16(d + (e * kRecV + v) * kRevBlock, rec + (long)i * kRecV + v);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float lam[5] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
  const int nst = (tot + kRevStage - 1) / kRevStage;
  fetch(0);
  for (int s = 0; s < nst; ++s) {
    fetch(s + 1);  // (empty past the last stage)
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    const float4* d = sh + (s & 1) * (kRevStage * kRecV * kRevBlock);
    for (int e = 0; e < kRevStage; ++e) {
      const int i = tot - 1 - s * kRevStage - e;
      if (i < 0) break;
      const float4 v0 = d[(e * kRecV + 0) * kRevBlock], v1 = d[(e * kRecV + 1) * kRevBlock];
      const float4 v2 = d[(e * kRecV + 2) * kRevBlock], v3 = d[(e * kRecV + 3) * kRevBlock];
      const float4 v4 = d[(e * kRecV + 4) * kRevBlock], v5 = d[(e * kRecV + 5) * kRevBlock];
      const float k0[5] = {v2.z, v2.w, v3.x, v3.y, v3.z};
      const float k1[5] = {v3.w, v4.x, v4.y, v4.z, v4.w};
      // (rounded by itself: fused into the sum in its place or one of the gains'
      // products, as the compiler chooses, the gradient would hang on that choice)
      float a0 = __fmul_rn(w2, v1.z), a1 = __fmul_rn(w2, v1.w);
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        a0 += k0[j] * lam[j];
        a1 += k1[j] * lam[j];
      }
      // (a step without an update has k = g = 0 here and no gradient)
      rec[(long)i * kRecV] = make_float4(v2.x * a0 + v2.y * a1, a0, a1, 0.0f);
      lam[0] -= a0;
      lam[1] -= a1;
      {
        const float l0 = lam[0], l1 = lam[1], l2 = lam[2];
        lam[2] = l2 + v0.x * l0 + v0.z * l1;
        lam[3] = lam[3] + v0.w * l1;
        lam[4] = lam[4] + v0.y * l0 + v1.x * l1 + v1.y * l2;
      }
      {
        const float l0 = lam[0], l1 = lam[1], l2 = lam[2];
        lam[0] = v5.x * l0 + v5.y * l1 + v5.z * l2;
        lam[2] = v5.w * l2;
      }
    }
  }
}

// Scatter of the gradients through the spline weights, one warp per track.  Its
// lanes first lay out 32 clusters' weights, cell and gradient in shared memory;
// then the warp takes the clusters in track order, each lane holding two of the
// cell's 64 control points for the three components.  A track stays about ten
// clusters in one cell, so the lanes sum in registers and add to the FP64
// accumulators only where the cell changes.  Those sums are kept in three floats
// (tf_add_product: finer than FP64 up to a track's 160 clusters): this GPU's FP64
// rate is 1/60 of its FP32 rate, and 192 FP64 operations per cluster would cost
// more than the whole sweep.  (Against float pairs, which fall short of FP64, the
// adjoint of 3.1e5 tracks takes 14.1 instead of 11.8 ms.)  Clusters whose gradients
// leave the range in which that holds (kSumLow, kSumHigh; infinities and NaN) are
// added term by term in FP64.  kShared: the block's accumulators lie in shared
// memory; a map too large for that has them in the block's partial sums in global
// memory.
constexpr int kScatWarps = 16;
constexpr int kScatF = 16;  // floats per staged cluster: wz[4], wr[4], wp[4], g[3], cell
constexpr unsigned kSumLow = (127u - 40u) << 23;    // 2^-40: 2^-149 is 2^-109 of the largest
constexpr unsigned kSumHigh = (127u + 100u) << 23;  // 2^100: 160 terms do not overflow

template <bool kShared>
__global__ void __launch_bounds__(32 * kScatWarps) k_refit_scatter(RefitDev R, KParams P,
                                                                   const int* steps3, int t0,
                                                                   int tn) {
  extern __shared__ double scat_sh[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* part = R.gpart + (long)blockIdx.x * R.ncoef;
  double* gacc = kShared ? scat_sh : part;
  float* st = (float*)(scat_sh + (kShared ? R.ncoef : 0)) + (long)warp * 32 * kScatF;
  if (kShared || t0 == 0)
    for (int i = threadIdx.x; i < R.ncoef; i += blockDim.x) gacc[i] = t0 == 0 ? 0.0 : part[i];
  __syncthreads();
  const MapDev M = R.map;
  const int la = lane >> 3, lb = (lane >> 1) & 3, lh = 2 * (lane & 1);  // z, r, first phi point
  const int nw = gridDim.x * (blockDim.x >> 5);
  const int ncomp = M.nz * M.nr * M.nphi;
  for (int q = blockIdx.x * (blockDim.x >> 5) + warp; q < tn; q += nw) {
    const int t = t0 + q;
    if (!R.ok[t]) continue;
    const int o0 = R.offset[t], ns = R.offset[t + 1] - o0;
    const int n3 = steps3[t];
    const float z0 = R.z0[t];
    const float4* rec = adj_rec(R, q);
    float hi[6], mid[6], lo[6];  // [component][point]
    int cell = -1;
    auto point = [&](int c, int e) {  // the lane's control point e of cell c
      const int zr = c / M.nphi;      // (z, r) cell corner
      return ((zr / M.nr + la) * M.nr + (zr % M.nr + lb)) * M.nphi +
             phi_index(c % M.nphi, lh + e, M.nphi);
    };
    auto flush = [&]() {
      if (cell < 0) return;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int at = point(cell, e);
#pragma unroll
        for (int c = 0; c < 3; ++c)
          atomicAdd(&gacc[c * ncomp + at],
                    (double)hi[2 * c + e] + ((double)mid[2 * c + e] + (double)lo[2 * c + e]));
      }
    };
    for (int k0 = 0; k0 < ns; k0 += 32) {
      const int k = k0 + lane;
      unsigned gmax = 0u;  // largest magnitude of the gradients (as bits: NaN above infinity)
      if (k < ns) {
        const float2 yz = R.raw[o0 + k];
        const int w = __float_as_int(R.meas[o0 + k].w);
        const SplinePt sp = spline_point<true>(M, P, w >> 8, R.row_x[w & 0xFF], yz.x, yz.y - z0);
        // the three iterations' gradients, in the order of the reverse sweep
        float gx = 0.0f, gy = 0.0f, gz = 0.0f;
#pragma unroll
        for (int it = 2; it >= 0; --it) {
          const int j = it == 1 ? k : ns - 1 - k;
          if (it == 2 && j >= n3) continue;
          const float4 g = rec[((long)it * ns + j) * kRecV];
          gx += g.x;
          gy += g.y;
          gz += g.z;
        }
        float* d = st + lane * kScatF;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          d[i] = sp.wz[i];
          d[4 + i] = sp.wr[i];
          d[8 + i] = sp.wp[i];
        }
        d[12] = gx;
        d[13] = gy;
        d[14] = gz;
        gmax = max(__float_as_uint(fabsf(gx)),
                   max(__float_as_uint(fabsf(gy)), __float_as_uint(fabsf(gz))));
        // (phi_index wraps its argument, so the cell's phi can be wrapped here)
        const int ipw = ((sp.ip % M.nphi) + M.nphi) % M.nphi;
        d[15] = __int_as_float((sp.iz * M.nr + sp.ir) * M.nphi + ipw);
      }
      __syncwarp();
      gmax = __reduce_max_sync(0xffffffffu, gmax);
      const int m = gmax != 0u ? min(32, ns - k0) : 0;
      const bool wide = gmax < kSumLow || gmax >= kSumHigh;
      for (int i = 0; i < m; ++i) {
        const float* d = st + i * kScatF;
        const int c = __float_as_int(d[15]);
        const float wzr = d[la] * d[4 + lb];
        if (wide) {
#pragma unroll 1
          for (int eg = 0; eg < 6; ++eg) {
            const int e = eg & 1, g = eg >> 1;
            if (d[12 + g] != 0.0f)
              atomicAdd(&gacc[g * ncomp + point(c, e)],
                        (double)(wzr * d[8 + lh + e]) * (double)d[12 + g]);
          }
          continue;
        }
        if (c != cell) {
          flush();
          cell = c;
#pragma unroll
          for (int e = 0; e < 6; ++e) hi[e] = mid[e] = lo[e] = 0.0f;
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float w = wzr * d[8 + lh + e];
#pragma unroll
          for (int g = 0; g < 3; ++g)
            tf_add_product(hi[2 * g + e], mid[2 * g + e], lo[2 * g + e], w, d[12 + g]);
        }
      }
      __syncwarp();
    }
    flush();
  }
  if (kShared) {
    __syncthreads();
    for (int i = threadIdx.x; i < R.ncoef; i += blockDim.x) part[i] = gacc[i];
  }
}

// Sum of the blocks' partial gradients in a fixed order: eight threads per
// coefficient, each over every eighth block, then the eight sums in turn.
__global__ void __launch_bounds__(256) k_grad_reduce(RefitDev R) {
  __shared__ double sh[8][32];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + x;
  double s = 0.0;
  if (i < R.ncoef)
    for (int b = y; b < R.gblocks; b += 8) s += R.gpart[(long)b * R.ncoef + i];
  sh[y][x] = s;
  __syncthreads();
  if (y == 0 && i < R.ncoef) {
    for (int k = 1; k < 8; ++k) s += sh[k][x];
    R.dl_dmap[i] = (float)s;
  }
}

}  // namespace

int map_pack(const MapDev& M, float4* c4, cudaStream_t s) {
  k_map_pack<<<blocks_for((long)M.nz * M.nr * M.nphi, 256), 256, 0, s>>>(M, c4);
  return 1;
}

template <bool kMap>
static void refit_passes(RefitDev& R, const KParams& P, int* steps3, unsigned g, int sms,
                         cudaStream_t s) {
  k_refit_iter<0, kMap><<<g, 128, 0, s>>>(R, P, steps3,
                                          resident_lanes<k_refit_iter<0, kMap>>(128, 0, g, sms));
  k_refit_iter<1, kMap><<<g, 128, 0, s>>>(R, P, steps3,
                                          resident_lanes<k_refit_iter<1, kMap>>(128, 0, g, sms));
  k_refit_iter<2, kMap><<<g, 128, 0, s>>>(R, P, steps3,
                                          resident_lanes<k_refit_iter<2, kMap>>(128, 0, g, sms));
}

int refit_forward(RefitDev& R, const KParams& P, int* steps3, int sms, cudaStream_t s) {
  if (R.n_tracks <= 0) return 0;
  // (no more blocks than there are tracks for)
  const unsigned g = (unsigned)min((long)sms * 4, (long)blocks_for(R.n_tracks, 32));
  k_refit_prep<<<(unsigned)min((long)sms * 16, (long)blocks_for(R.n_tracks, 8)), 256, 0, s>>>(
      R, P, steps3);
  k_refit_order<<<(unsigned)min((long)sms * 4, (long)blocks_for(R.n_tracks, kOrdChunk)), kBlock, 0,
                  s>>>(R, P);
  k_refit_start<<<g, 128, 0, s>>>(R, P, resident_lanes<k_refit_start>(128, 0, g, sms));
  if (R.map.on) refit_passes<true>(R, P, steps3, g, sms, s);
  else refit_passes<false>(R, P, steps3, g, sms, s);
  return 6;
}

int refit_backward(RefitDev& R, const KParams& P, const int* steps3, int sms, cudaStream_t s) {
  (void)sms;
  const size_t rev = sizeof(float4) * 2 * kRevStage * kRecV * kRevBlock;
  const size_t acc = sizeof(double) * (size_t)R.ncoef;
  const size_t stage = sizeof(float) * 32 * kScatF;  // per warp
  // accumulators in shared memory beside the staging of at least four warps
  // (the 18 x 16 x 20 map's 138 KB leave room for all sixteen)
  int warps = kScatWarps;
  bool shared = true;
  while (warps > 4 && acc + warps * stage > (size_t)R.smem_max) --warps;
  if (acc + warps * stage > (size_t)R.smem_max) {
    shared = false;
    warps = kScatWarps;
  }
  const size_t scat = (shared ? acc : 0) + warps * stage;
  // (process-wide attributes: the same values in every call, whatever its map, so that
  // no other context's thread lowers a limit between this call's set and launch)
  cudaFuncSetAttribute(k_refit_reverse, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rev);
  cudaFuncSetAttribute(k_refit_scatter<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       R.smem_max);
  int k = 0;
  long t0 = 0;
  do {
    const int tn = (int)min(R.n_tracks - t0, (long)R.chunk);
    if (tn > 0) {
      k_refit_replay<<<blocks_for((long)tn * 3 * kCkptSeg, 128), 128, 0, s>>>(R, P, steps3,
                                                                              (int)t0, tn);
      k_refit_reverse<<<blocks_for(tn, kRevBlock), kRevBlock, rev, s>>>(R, steps3, (int)t0, tn);
      k += 2;
    }
    if (shared)
      k_refit_scatter<true><<<R.gblocks, 32 * warps, scat, s>>>(R, P, steps3, (int)t0, tn);
    else
      k_refit_scatter<false><<<R.gblocks, 32 * warps, scat, s>>>(R, P, steps3, (int)t0, tn);
    ++k;
    t0 += R.chunk;
  } while (t0 < R.n_tracks);
  k_grad_reduce<<<blocks_for(R.ncoef, 32), 256, 0, s>>>(R);
  return k + 1;
}

int stage_sector_refit(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  const int nb_tl = (int)blocks_for(F.cap_tl, kBlock);
  k_acc_count<<<nb_tl, kBlock, 0, s>>>(F);
  k_scan_partials<<<1, 1024, 0, s>>>(F.scan_tmp, nb_tl, &F.cnt->n_tracks);
  k_acc_write<<<nb_tl, kBlock, 0, s>>>(F);
  k_order_scatter<<<sms * 4, kBlock, 0, s>>>(F.st_obucket, F.st_oslot, F.st_ord_cnt,
                                             &F.cnt->n_tracks, F.cap_tl, &F.cnt->err, F.st_order);
  k_st_gather<<<sms * 8, kBlock, 0, s>>>(F, P);
  const unsigned g = persistent_grid(F.lc, kLSectorRefit, sms);
  const int b = F.lc.block[kLSectorRefit];
  k_sector_refit<<<g, b, 0, s>>>(F, P, resident_lanes<k_sector_refit>(b, 0, g, sms));
  return 6;
}

int stage_merge(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  const int nb_tl = (int)blocks_for(F.cap_tl, kBlock);
  k_sector_zrange<<<P.n_sectors, 256, 0, s>>>(F, P);
  k_ie_hist<<<sms * 8, kBlock, 0, s>>>(F, P);
  int k = 2;
  k += scan_exclusive(F.ie_cnt, F.ie_first, (long)P.n_sectors * P.n_rows * kMergeZ + 1,
                      F.scan_tmp, s);
  k_ie_scatter<<<sms * 8, kBlock, 0, s>>>(F);
  {
    const unsigned grid = persistent_grid(F.lc, kLMerge, sms);
    const int blk = F.lc.block[kLMerge];
    switch (F.lc.lanes[kLMerge]) {
      case 32: k_merge_best<32><<<grid, blk, 0, s>>>(F, P); break;
      case 16: k_merge_best<16><<<grid, blk, 0, s>>>(F, P); break;
      case 8: k_merge_best<8><<<grid, blk, 0, s>>>(F, P); break;
      case 4: k_merge_best<4><<<grid, blk, 0, s>>>(F, P); break;
      default: k_merge_best<1><<<grid, blk, 0, s>>>(F, P); break;
    }
  }
  k_merge_link<<<sms * 8, kBlock, 0, s>>>(F);
  if (P.ac_merge) {
    k_cross_best<<<sms * 8, kBlock, 0, s>>>(F, P);
    k_cross_link<<<sms * 8, kBlock, 0, s>>>(F);
    k += 2;
  }
  k_head_count<<<nb_tl, kBlock, 0, s>>>(F);
  k_scan_partials<<<1, 1024, 0, s>>>(F.scan_tmp, nb_tl, &F.cnt->n_merged);
  k_head_write<<<nb_tl, kBlock, 0, s>>>(F, P);
  const int nb_ft = (int)blocks_for(F.cap_ft, kBlock);
  k_looper_count<<<nb_ft, kBlock, 0, s>>>(F);
  k_scan_partials<<<1, 1024, 0, s>>>(F.scan_tmp, nb_ft, &F.cnt->n_loopers);
  k_looper_write<<<nb_ft, kBlock, 0, s>>>(F);
  return k + 9;
}

// The fit kernels' variants: with a correction map or without, with the Phase
// III rows or without (the common form carries neither's code nor registers).
template <bool kMap>
int fit12(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  const unsigned g = persistent_grid(F.lc, kLFit12, sms);
  const int b = F.lc.block[kLFit12];
  k_fit_stations<kMap><<<sms * 8, kBlock, 0, s>>>(F, P, F.map);
  k_fit_order<<<sms * 4, kBlock, 0, s>>>(F);
  if (P.ext_rows > 0) {
    k_fit1<kMap, true><<<g, b, 0, s>>>(F, P, F.map, resident_lanes<k_fit1<kMap, true>>(b, 0, g, sms));
    k_fit2<kMap, true><<<g, b, 0, s>>>(F, P, F.map, resident_lanes<k_fit2<kMap, true>>(b, 0, g, sms));
  } else {
    k_fit1<kMap, false><<<g, b, 0, s>>>(F, P, F.map, resident_lanes<k_fit1<kMap, false>>(b, 0, g, sms));
    k_fit2<kMap, false><<<g, b, 0, s>>>(F, P, F.map, resident_lanes<k_fit2<kMap, false>>(b, 0, g, sms));
  }
  k_inner_cand<kMap><<<sms * 8, kBlock, 0, s>>>(F, P, F.map);
  return 5;  // the station lists, the order, iterations 1 and 2, the candidate search
}

int stage_fit12(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  return F.map.on ? fit12<true>(F, P, sms, s) : fit12<false>(F, P, sms, s);
}

int stage_ambiguity2(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  int k = 0;
  for (int r = 0; r < P.cand_k; ++r) {
    k_amb_bid<<<sms * 8, kBlock, 0, s>>>(F, P, r);
    if (r + 1 < P.cand_k) k_amb_resolve<false, false><<<sms * 8, kBlock, 0, s>>>(F, P, F.map, r);
    else if (F.map.on) k_amb_resolve<true, true><<<sms * 8, kBlock, 0, s>>>(F, P, F.map, r);
    else k_amb_resolve<true, false><<<sms * 8, kBlock, 0, s>>>(F, P, F.map, r);
    k += 2;
  }
  return k;
}

template <bool kMap, bool kExt>
int fit3(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  const unsigned g = persistent_grid(F.lc, kLFit3, sms);
  const int b = F.lc.block[kLFit3];
  k_fit3<kMap, kExt><<<g, b, 0, s>>>(F, P, F.map, resident_lanes<k_fit3<kMap, kExt>>(b, 0, g, sms));
  return 1;
}

int stage_fit3(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  if (P.ext_rows > 0)
    return F.map.on ? fit3<true, true>(F, P, sms, s) : fit3<false, true>(F, P, sms, s);
  return F.map.on ? fit3<true, false>(F, P, sms, s) : fit3<false, false>(F, P, sms, s);
}

int stage_output(FrameDev& F, const KParams& P, int sms, cudaStream_t s) {
  const int nb = (int)blocks_for(F.cap_ft, kBlock);
  k_out_count<<<nb, kBlock, 0, s>>>(F, P);
  k_out_scan<<<1, 1024, 0, s>>>(F, nb);
  k_out_write<<<nb, kBlock, 0, s>>>(F, P);
  k_out_lists<<<sms * 8, kBlock, 0, s>>>(F);
  k_out_attach<<<sms * 8, kBlock, 0, s>>>(F, P);
  return 5;
}

}  // namespace TPC_NS
}  // namespace tpc
