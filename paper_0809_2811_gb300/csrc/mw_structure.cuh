// mw_structure.cuh -- structure analysis of the current positions (Sec. II.C):
// the pair histogram behind the radial distribution function g(r) and the
// angle histogram behind the angular distribution function (the angles at an
// atom between its n_c nearest neighbours).  Both read a neighbour list built
// at the current positions, so every pair within the list radius is in it.
// A group of lanes per centre; counts of the block's first and last box are
// summed in shared memory (32-bit) and added to the per-box 64-bit histogram
// once per block, other boxes (small boxes only) go to global memory directly.
// Both are bound by latency (dependent gathers, and per centre the search for
// its nearest); on two boxes of 32768 atoms the pair histogram takes 15 us
// and the angle histogram (n_c = 8) 41 us (18 and 73 us with one thread per
// centre walking its row and sorting in local memory).
#pragma once

#include "mw_device.cuh"

namespace mw {

constexpr int kSThreads = 128;
constexpr int kAdfMax = 16;  // largest n_c of the angle histogram

struct BlockHist {
  unsigned* sh;  // [2][nbins]
  unsigned long long* glob;  // [nbox][nbins]
  int nbins, b_first, b_last;

  // the block's centres: i0 ... i0 + count - 1
  __device__ void begin(const Dev& d, unsigned* s, int nb, unsigned long long* g, int i0, int count) {
    sh = s;
    glob = g;
    nbins = nb;
    b_first = (int)d.q[i0].w;
    b_last = (int)d.q[min(i0 + count, d.N) - 1].w;
    for (int k = threadIdx.x; k < 2 * nbins; k += blockDim.x) sh[k] = 0u;
    __syncthreads();
  }
  __device__ void add(int b, int k, unsigned c) {
    if (b == b_first) atomicAdd(sh + k, c);
    else if (b == b_last) atomicAdd(sh + nbins + k, c);
    else atomicAdd(glob + (size_t)b * nbins + k, (unsigned long long)c);
  }
  __device__ void end() {
    __syncthreads();
    for (int k = threadIdx.x; k < nbins; k += blockDim.x) {
      if (sh[k]) atomicAdd(glob + (size_t)b_first * nbins + k, (unsigned long long)sh[k]);
      if (b_last != b_first && sh[nbins + k]) atomicAdd(glob + (size_t)b_last * nbins + k, (unsigned long long)sh[nbins + k]);
    }
  }
};

// r^2 of row entry s of a centre (row, qi, box bx), and its vector.
__device__ __forceinline__ float row_r2(const Dev& d, const uint4& qi, const Box& bx, int j, float& dx, float& dy, float& dz) {
  const uint4 qj = d.q[j];
  dx = fix_diff(qi.x, qj.x, bx.Lq[0]);
  dy = fix_diff(qi.y, qj.y, bx.Lq[1]);
  dz = fix_diff(qi.z, qj.z, bx.Lq[2]);
  return fmaf(dx, dx, fmaf(dy, dy, dz * dz));
}

// Pair histogram: every ordered pair (i, j), i != j, of one box with
// k dr <= r_ij < (k + 1) dr, k < nbins (nbins dr within the list radius).
constexpr int kPairLanes = 4;
constexpr int kPairCentres = kSThreads / kPairLanes;
__global__ void __launch_bounds__(kSThreads) k_pair_hist(Dev d, float inv_dr, float rmax2, int nbins,
                                                         unsigned long long* hist) {
  extern __shared__ unsigned s_hist[];
  const int i0 = (int)blockIdx.x * kPairCentres;
  BlockHist h;
  h.begin(d, s_hist, nbins, hist, i0, kPairCentres);
  const int i = i0 + (int)threadIdx.x / kPairLanes;
  if (i < d.N) {
    const uint4 qi = d.q[i];
    const Box& bx = d.box[qi.w];
    const int cnt = min(d.nbr_cnt[i], d.W);
    const int* row = d.nbr + (size_t)i * d.W;
#pragma unroll 4
    for (int s = (int)threadIdx.x % kPairLanes; s < cnt; s += kPairLanes) {
      float dx, dy, dz;
      const float r2 = row_r2(d, qi, bx, row[s], dx, dy, dz);
      if (r2 < rmax2) {
        const int k = (int)(sqrtf(r2) * inv_dr);
        if (k < nbins) h.add((int)qi.w, k, 1u);
      }
    }
  }
  h.end();
}

// Angle histogram: for each atom k its nc nearest neighbours (from the list;
// fewer than nc within the list radius is counted in *short_rows), the angle
// theta_ikj at k for every ordered pair i != j of them, binned over
// [0, 180] degrees (180 itself in the last bin).  kAngLanes lanes per centre:
// they hold the row's squared distances in shared memory, rank their own
// against all of them (ties by place in the row; rows longer than kAngRow pick
// the nc smallest one after the other, recomputing what is not held), and
// share the pairs of the nc nearest.
constexpr int kAngLanes = 8;
constexpr int kAngCentres = kSThreads / kAngLanes;
constexpr int kAngRow = 96;
__global__ void __launch_bounds__(kSThreads) k_angle_hist(Dev d, int nc, int nbins, float inv_w,
                                                          unsigned long long* hist, int* short_rows) {
  extern __shared__ unsigned s_hist[];
  __shared__ float s_r2[kAngCentres][kAngRow + 1];
  __shared__ float s_u[kAngCentres][kAdfMax][3];
  const int i0 = (int)blockIdx.x * kAngCentres;
  BlockHist h;
  h.begin(d, s_hist, nbins, hist, i0, kAngCentres);
  const int a = (int)threadIdx.x / kAngLanes, g = (int)threadIdx.x % kAngLanes;
  const int i = i0 + a;
  const bool valid = i < d.N;
  const unsigned group = ((1u << kAngLanes) - 1u) << (threadIdx.x & 31 & ~(kAngLanes - 1));  // this centre's lanes
  uint4 qi = make_uint4(0u, 0u, 0u, 0u);
  int cnt = 0;
  if (valid) {
    qi = d.q[i];
    cnt = min(d.nbr_cnt[i], d.W);
  }
  const Box& bx = d.box[qi.w];
  const int* row = d.nbr + (size_t)(valid ? i : 0) * d.W;
  float dx, dy, dz;
#pragma unroll 4
  for (int s = g; s < min(cnt, kAngRow); s += kAngLanes) s_r2[a][s] = row_r2(d, qi, bx, row[s], dx, dy, dz);
  __syncwarp();
  if (valid && cnt < nc) {
    if (g == 0) atomicAdd(short_rows, 1);
  } else if (valid) {
    auto place = [&](int m, int s) {  // row entry s is the centre's m-th nearest
      const float r2 = row_r2(d, qi, bx, row[s], dx, dy, dz);
      const float inv = rsqrtf(r2);
      s_u[a][m][0] = dx * inv;
      s_u[a][m][1] = dy * inv;
      s_u[a][m][2] = dz * inv;
    };
    // order of a candidate: (r^2, place in the row); r^2 >= 0, so its bits order like it
    if (cnt <= kAngRow) {  // ranks: each lane's candidates, four at a time, against all of the row
      for (int s0 = g; s0 < cnt; s0 += 4 * kAngLanes) {
        int rank[4] = {0, 0, 0, 0}, mine[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) mine[k] = s0 + k * kAngLanes < cnt ? __float_as_int(s_r2[a][s0 + k * kAngLanes]) : 0x7fffffff;
        for (int t = 0; t < cnt; ++t) {
          const int r = __float_as_int(s_r2[a][t]);
#pragma unroll
          for (int k = 0; k < 4; ++k) rank[k] += r - (t < s0 + k * kAngLanes ? 1 : 0) < mine[k] ? 1 : 0;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (s0 + k * kAngLanes < cnt && rank[k] < nc) place(rank[k], s0 + k * kAngLanes);
      }
    } else {  // long rows: the least above the last, nc times
      unsigned last_r = 0u;
      int last_s = -1;
      for (int m = 0; m < nc; ++m) {
        unsigned best_r = 0xffffffffu;
        int best_s = 0x7fffffff;
        for (int s = g; s < cnt; s += kAngLanes) {
          const unsigned r = __float_as_uint(s < kAngRow ? s_r2[a][s] : row_r2(d, qi, bx, row[s], dx, dy, dz));
          const bool above = r > last_r || (r == last_r && s > last_s);
          if (above && r < best_r) {  // (places ascend within a lane: the first of equals stays)
            best_r = r;
            best_s = s;
          }
        }
#pragma unroll
        for (int o = 1; o < kAngLanes; o <<= 1) {
          const unsigned r = __shfl_xor_sync(group, best_r, o);
          const int s = __shfl_xor_sync(group, best_s, o);
          if (r < best_r || (r == best_r && s < best_s)) {
            best_r = r;
            best_s = s;
          }
        }
        last_r = best_r;
        last_s = best_s;
        if (best_s % kAngLanes == g) place(m, best_s);
      }
    }
    __syncwarp(group);
    for (int p = g; p < nc * (nc - 1) / 2; p += kAngLanes) {  // pair p of p = y (y - 1) / 2 + x, x < y
      int y = (int)(0.5f + sqrtf(0.25f + 2.0f * (float)p));
      if (y * (y - 1) / 2 > p) --y;
      if (y * (y + 1) / 2 <= p) ++y;
      const int x = p - y * (y - 1) / 2;
      const float* u = s_u[a][x];
      const float* w = s_u[a][y];
      float c = fmaf(u[0], w[0], fmaf(u[1], w[1], u[2] * w[2]));
      c = fminf(1.0f, fmaxf(-1.0f, c));
      const float th = acosf(c) * 57.29577951308232f;
      const int k = min(nbins - 1, (int)(th * inv_w));
      h.add((int)qi.w, k, 2u);  // the ordered pairs (x, y) and (y, x)
    }
  }
  h.end();
}

}  // namespace mw
