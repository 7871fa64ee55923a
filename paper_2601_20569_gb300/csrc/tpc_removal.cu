// Online cluster removal (Sec. 4) on the tracks of the last tracking call.
//
// Clusters inside a protective tube around physics tracks are kept; of the
// others, those inside a removal tube around secondary looper legs and
// around very-low-pT tracks are flagged for removal; the clusters of the
// tracklets a physics track was built from (its seeding history) are
// protected too.  The section gives the rules in words; the readings:
// * very low pT: |q/pT| at the innermost cluster above qpt;
// * looper legs: two looper tracks (|q/pT| > looper_qpt) of one side whose
//   |q/pT| differ by at most leg_dq relative, whose tan(lambda) are opposite
//   within leg_dtgl (legs flown inwards are parametrised outwards) and whose
//   circle centres in global coordinates lie within leg_dc; |z| grows along
//   the looper and side * z_measured differs from it by one constant of the
//   collision, so a leg linked to one with a smaller side * z at the
//   innermost cluster is a secondary leg; its parent is the first such leg
//   (smallest (side * z, key), the track key breaking exact ties);
// * tubes follow the track's clusters, with the linear interpolation from
//   the lower-row cluster on the rows between two consecutive clusters of one
//   sector; protection 1 = a wide protective and a narrow removal tube;
//   protection 2 (mode 2) scales them on the innermost rows, near the sector
//   edge and where the occupancy around the centre is high.
// Every decision is an integer or a comparison of FP32 values computed in the
// same order as the strict CPU oracle; flags are combined with atomicOr, so
// the result does not depend on the order of the threads.
#include <cuda_runtime.h>

#include "tpc_internal.h"
#include "tpc_kernels.h"
#include "tpc_util.cuh"

namespace tpc {
namespace TPC_NS {
namespace {

constexpr float kCrHalfRange = 256.0f;  // circle centres binned over [-256, 256) cm per axis

// Centre bin of a circle centre (clamped: centres outside the range share the
// edge bins, which keeps any two centres within one bin width in adjacent bins).
__device__ __forceinline__ int centre_bin(float c, const RemovalParams& R) {
  return min(R.nbx - 1, max(0, (int)floorf((c + kCrHalfRange) * R.inv_cell)));
}

__device__ __forceinline__ int out_count(const FrameDev& F) { return F.cnt->n_out; }

// Class, looper flag, leg order key and circle centre of every output track;
// loopers are counted per (side block, centre bin).
__global__ void k_cr_tracks(FrameDev F, KParams P, RemovalParams R) {
  const int nt = out_count(F);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
    const float* o = F.out_par + (long)t * 5;
    const int s = F.out_sector[t];
    const float q = o[4];
    const float side = (s % R.nsec_frame) < R.half ? 1.0f : -1.0f;
    F.cr_zk[t] = side * o[1];
    F.cr_cls[t] = fabsf(q) > R.qpt ? 1 : 0;
    F.cr_parent[t] = -1;
    // the curvature centre lies 1/kappa along the left normal of the direction
    const float rk = 1.0f / (P.kb * q);
    const float sn = o[2];
    const float cs = sqrtf(1.0f - sn * sn);
    const float xc = F.out_x[t] - sn * rk, yc = o[0] + cs * rk;
    const int a = s % 18;
    const float cx = xc * R.sec_cos[a] - yc * R.sec_sin[a];
    const float cy = xc * R.sec_sin[a] + yc * R.sec_cos[a];
    F.cr_cx[t] = cx;
    F.cr_cy[t] = cy;
    if (P.looper_qpt > 0.0f && fabsf(q) > P.looper_qpt) {
      const int b = ((s / R.half) * R.nbx + centre_bin(cy, R)) * R.nbx + centre_bin(cx, R);
      atomicAdd(&F.cr_bin_cnt[b], 1);
    }
  }
}

__device__ __forceinline__ int cr_bin(const FrameDev& F, const RemovalParams& R, int t) {
  return ((F.out_sector[t] / R.half) * R.nbx + centre_bin(F.cr_cy[t], R)) * R.nbx +
         centre_bin(F.cr_cx[t], R);
}

__device__ __forceinline__ bool is_looper(const FrameDev& F, const KParams& P, int t) {
  return P.looper_qpt > 0.0f && fabsf(F.out_par[(long)t * 5 + 4]) > P.looper_qpt;
}

// Loopers into their bins (bin order is irrelevant: the leg search takes a
// minimum over the whole neighbourhood), as records of what the search tests: it
// walks them in bin order, where six gathers per candidate took 95 us on a
// 4e6-cluster frame.
__global__ void k_cr_scatter(FrameDev F, KParams P, RemovalParams R) {
  const int nt = out_count(F);
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nt; t += gridDim.x * blockDim.x) {
    if (!is_looper(F, P, t)) continue;
    const int b = cr_bin(F, R, t);
    const int at = F.cr_bin_first[b] + atomicSub(&F.cr_bin_cnt[b], 1) - 1;
    const float* o = F.out_par + (long)t * 5;
    F.cr_rec[2 * (long)at] = make_float4(o[4], o[3], F.cr_cx[t], F.cr_cy[t]);
    F.cr_rec[2 * (long)at + 1] =
        make_float4(F.cr_zk[t], __int_as_float(F.out_key[t]), __int_as_float(t), 0.0f);
  }
}

// Secondary legs: the first earlier leg among the loopers of the 3 x 3
// neighbouring centre bins (bins are at least leg_dc wide).
__global__ void k_cr_legs(FrameDev F, KParams P, RemovalParams R) {
  const int nt = out_count(F);
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < nt; a += gridDim.x * blockDim.x) {
    if (!is_looper(F, P, a)) continue;
    const float qa = F.out_par[(long)a * 5 + 4], ta = F.out_par[(long)a * 5 + 3];
    const float xa = F.cr_cx[a], ya = F.cr_cy[a], za = F.cr_zk[a];
    const float aa = fabsf(qa);
    const int ka = F.out_key[a];
    const int b0 = cr_bin(F, R, a);
    const int xb = b0 % R.nbx, yb = (b0 / R.nbx) % R.nbx;
    int best = -1, bk = 0;
    float bz = 0.0f;
    for (int e = -1; e <= 1; ++e) {
      if (yb + e < 0 || yb + e >= R.nbx) continue;
      // the three x bins of centre row yb + e are contiguous
      const int x0 = max(0, xb - 1), x1 = min(R.nbx - 1, xb + 1);
      const int row0 = b0 - xb + e * R.nbx;
      const int lo = F.cr_bin_first[row0 + x0], hi = F.cr_bin_first[row0 + x1 + 1];
      for (int j = lo; j < hi; ++j) {
        const float4 v = F.cr_rec[2 * (long)j];
        const float qb = v.x;
        if ((qa > 0.0f) == (qb > 0.0f)) continue;
        const float ab = fabsf(qb);
        const float mx = aa > ab ? aa : ab;
        if (!(fabsf(aa - ab) <= R.leg_dq * mx)) continue;
        if (!(fabsf(ta + v.y) <= R.leg_dtgl)) continue;
        const float dx = xa - v.z, dy = ya - v.w;
        if (!(dx * dx + dy * dy <= R.leg_dc * R.leg_dc)) continue;
        const float4 u = F.cr_rec[2 * (long)j + 1];
        const int b = __float_as_int(u.z);  // (a itself fails the charge test)
        const float zb = u.x;
        const int kb = __float_as_int(u.y);
        if (!(zb < za || (zb == za && kb < ka))) continue;
        if (best < 0 || zb < bz || (zb == bz && kb < bk)) {
          best = b;
          bz = zb;
          bk = kb;
        }
      }
    }
    if (best >= 0) {
      F.cr_parent[a] = best;
      F.cr_cls[a] = 2;
    }
  }
}

// One tube cross-section: the clusters of batch row rr within h of (yc, zc).
// Where protection 2 depends on the occupancy, one scan of the window that
// covers both the occupancy window and the larger of the two possible tubes
// counts the occupancy and marks the clusters of both tubes.  The window's whole z
// strips are one contiguous run of the sorted order, walked in one loop that the
// lanes of a warp run together, with the tubes as bit masks; where it holds
// more than 32 clusters, the bins of the window are walked strip by strip (and
// again once h is known).  (Strip by strip with a list in local memory for all:
// 0.60 ms on a 4e6-cluster frame.)
__device__ __forceinline__ void cr_tube(const FrameDev& F, const KParams& P,
                                        const RemovalParams& R, int rr, float yc, float zc,
                                        bool protect) {
  const int r = rr % P.n_rows;
  const RowGrid g = F.rows[rr];
  const float h0 = protect ? R.protect : R.remove;
  const float fac = protect ? R.p2_grow : R.p2_shrink;
  const unsigned bit = protect ? 1u : 4u;
  const float hg = h0 * fac, w = R.occ_w;
  bool grown = false, by_occ = false;  // half-width hg instead of h0; by the occupancy
  if (R.mode >= 2) {
    if (r < P.inner_rows || fabsf(yc) > F.row_x[r] * P.tan_half - R.edge) grown = true;
    else by_occ = true;
  }
  const float wb = by_occ ? fmaxf(w, fmaxf(h0, hg)) : grown ? hg : h0;
  if (g.ncl == 0 || !(yc - wb <= yc + wb) || !(zc - wb <= zc + wb)) return;
  const int iz0 = bin_of(zc - wb, g.z0, g.invDz, g.nZ), iz1 = bin_of(zc + wb, g.z0, g.invDz, g.nZ);
  const int lo = F.bin_first[g.bin0 + iz0 * g.nY];
  const int n = F.bin_first[g.bin0 + (iz1 + 1) * g.nY] - lo;
  if (n <= 32) {
    int occ = 0;
    unsigned in0 = 0u, ing = 0u;  // within h0, within hg
    for (int c = 0; c < n; ++c) {
      const float2 pk = F.syz[lo + c];
      const float dy = fabsf(pk.x - yc), dz = fabsf(pk.y - zc);
      if (dy <= w && dz <= w) ++occ;
      if (dy <= h0 && dz <= h0) in0 |= 1u << c;
      if (dy <= hg && dz <= hg) ing |= 1u << c;
    }
    if (by_occ) grown = occ > R.occ_max;
    for (unsigned m = grown ? ing : in0; m; m &= m - 1u)
      atomicOr(&F.cr_flags[lo + __ffs(m) - 1], bit);
    return;
  }
  if (by_occ) {
    int occ = 0;
    for_window(F.bin_first, g, yc - w, yc + w, zc - w, zc + w, [&](int k) {
      const float2 pk = F.syz[k];
      if (fabsf(pk.x - yc) <= w && fabsf(pk.y - zc) <= w) ++occ;
    });
    grown = occ > R.occ_max;
  }
  const float h = grown ? hg : h0;
  for_window(F.bin_first, g, yc - h, yc + h, zc - h, zc + h, [&](int k) {
    const float2 pk = F.syz[k];
    if (fabsf(pk.x - yc) <= h && fabsf(pk.y - zc) <= h) atomicOr(&F.cr_flags[k], bit);
  });
}

// Tubes of every output track and the seeding history of the physics ones.
// A track's tube cross-sections do not depend on one another: one warp per
// track; the cross-sections of 32 clusters and of the gap rows between them are
// dealt out to the lanes (a lane per cluster that walked its gap rows made the
// warp wait for the longest gap), then the lanes take the rows of each seeding
// tracklet.
// (One thread per track, walking its clusters in turn, was bound by that serial
// chain of window scans: 1.06 ms for the 4,600 tracks of an event.)
__global__ void k_cr_tubes(FrameDev F, KParams P, RemovalParams R) {
  const int nf = min(F.cnt->n_merged, (int)F.cap_ft);
  const int NR = P.n_rows;
  const int lane = threadIdx.x & 31;
  const int nw = gridDim.x * (blockDim.x >> 5);
  for (int f = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); f < nf; f += nw) {
    const int t = F.ft_outidx[f];
    if (t < 0) continue;
    const bool protect = F.cr_cls[t] == 0;
    const int n = F.ft_n[f];
    if (n <= 0) continue;
    const int* used = F.ft_used + (long)f * kMaxRows;
    for (int i0 = 0; i0 < n; i0 += 32) {
      // the lane's cluster and the next one; g rows lie between them where they
      // share a sector
      const int i = i0 + lane;
      const int c = i < n ? used[i] : -1, d = i + 1 < n ? used[i + 1] : -1;
      const int crr = c >= 0 ? F.srow[c] : 0, drr = d >= 0 ? F.srow[d] : -1;
      const float2 pc = c >= 0 ? F.syz[c] : make_float2(0.0f, 0.0f);
      const float2 pd = d >= 0 ? F.syz[d] : make_float2(0.0f, 0.0f);
      const bool cl = crr < drr;  // interpolate from the lower-row cluster
      const int rlo = cl ? crr : drr, rhi = cl ? drr : crr;
      const float2 plo = cl ? pc : pd, phi = cl ? pd : pc;
      const int g = d >= 0 && drr / NR == crr / NR ? max(0, rhi - rlo - 1) : 0;
      const int cnt = c >= 0 ? 1 + g : 0;
      int inc = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      const int total = __shfl_sync(0xffffffffu, inc, 31);
      for (int q0 = 0; q0 < total; q0 += 32) {
        const int q = q0 + lane;
        int L = 0;  // the lane whose cluster or gap row item q is: first with inc > q
#pragma unroll
        for (int st = 16; st >= 1; st >>= 1) {
          const int v = __shfl_sync(0xffffffffu, inc, L + st - 1);
          if (v <= q) L += st;
        }
        const int e = q - __shfl_sync(0xffffffffu, inc - cnt, L);  // 0: the cluster itself
        const int lrr = __shfl_sync(0xffffffffu, crr, L);
        const int llo = __shfl_sync(0xffffffffu, rlo, L), lhi = __shfl_sync(0xffffffffu, rhi, L);
        const float cx = __shfl_sync(0xffffffffu, pc.x, L), cy = __shfl_sync(0xffffffffu, pc.y, L);
        const float lx = __shfl_sync(0xffffffffu, plo.x, L), ly = __shfl_sync(0xffffffffu, plo.y, L);
        const float hx = __shfl_sync(0xffffffffu, phi.x, L), hy = __shfl_sync(0xffffffffu, phi.y, L);
        if (q >= total) continue;
        const float fr = (float)e / (float)(lhi - llo);
        cr_tube(F, P, R, e == 0 ? lrr : llo + e, e == 0 ? cx : lx + (hx - lx) * fr,
                e == 0 ? cy : ly + (hy - ly) * fr, protect);
      }
    }
    if (!protect) continue;
    for (int sg = F.ft_head[f]; sg >= 0; sg = F.st_next[sg]) {
      const int ti = F.st_tl[sg];
      const int* H = F.tl_hits + (long)ti * kMaxRows;
      const int rhi = F.tl_rhi[ti];
      for (int r = F.tl_rlo[ti] + lane; r <= rhi; r += 32)
        if (H[r] >= 0) atomicOr(&F.cr_flags[H[r]], 2u);
    }
  }
}

// Removed = in a removal tube, neither protected nor history; flags out in
// input order, removed clusters counted.
__global__ void k_cr_final(FrameDev F) {
  for (long k = (long)blockIdx.x * blockDim.x + threadIdx.x; k < F.n;
       k += (long)gridDim.x * blockDim.x) {
    unsigned fl = F.cr_flags[k];
    const bool rem = (fl & 4u) && !(fl & 3u);
    if (rem) fl |= 8u;
    F.cr_out[F.sid[k]] = (uint8_t)fl;
    const unsigned m = __ballot_sync(__activemask(), rem);
    if (rem && (threadIdx.x & 31) == __ffs(m) - 1) atomicAdd(&F.cnt->n_removed, __popc(m));
  }
}

}  // namespace

int cluster_removal(FrameDev& F, const KParams& P, const RemovalParams& R, int nblk, int sms,
                    cudaStream_t s) {
  const int nbins = nblk * R.nbx * R.nbx;
  const int g = sms * 8;
  k_cr_tracks<<<g, kBlock, 0, s>>>(F, P, R);
  int k = 1 + scan_exclusive(F.cr_bin_cnt, F.cr_bin_first, nbins + 1, F.scan_tmp, s);
  k_cr_scatter<<<g, kBlock, 0, s>>>(F, P, R);
  k_cr_legs<<<g, kBlock, 0, s>>>(F, P, R);
  k_cr_tubes<<<g, kBlock, 0, s>>>(F, P, R);
  k_cr_final<<<g, kBlock, 0, s>>>(F);
  return k + 4;
}

}  // namespace TPC_NS
}  // namespace tpc
