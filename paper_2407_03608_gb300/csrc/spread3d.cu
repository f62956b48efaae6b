// Steps (1) + (2a) of Sec. 4.2 in three dimensions, on the box grids of fft3d.cu: spread
// c_k,i = w_k(x_i) alpha_i onto all Chebyshev channels k at once, accumulating in registers.
//
// Output-stationary tiles of 32 columns (last axis) by 2 RPW rows by 4 planes.  Warp w of the
// CTA owns plane w / 2 and the band of RPW rows w % 2; its lanes form four groups of eight,
// and group g owns the strip of columns 8g .. 8g + 7.  Each lane keeps the RPW x C sums of its
// column in registers.  For every (warp, group) pair the CTA builds the ordered list of the
// points whose support meets its cells, so each group walks only its own list and the four
// groups of a warp spread four different points per instruction.
//
// The CTA scans the points of the bins that can reach the tile (one per thread), compacts the
// ones that do into a queue in sorted order, and works off the queue kSlots points at a time:
// their kernel values per axis and w_k alpha go to shared memory, ballots fill the 32 lists.
// The order, and so the summation order, is fixed (results are reproducible bit for bit).
// Every grid value is written once; tiles no point can reach are never launched and stay zero.
//
// FP32 sums are kept as pairs of channels, one packed multiply-add each (the same roundings), and
// in two words: every kFold list steps the running sum joins the total by TwoSum (ff64.h), and its
// rounding error starts the next running sum.  So a cell's error is that of kFold additions
// however many points reach it.  Relative l2 error of an FP32 product to the float64 plan on the
// same grid, 2e5 points of one sign in a tenth of the box (8600 contributions a cell): 1.05e-6 with
// the general kernel's fixed-point sums, 7.7e-7 here, 7.9e-6 with one word a sum; 2e6 uniform points
// at nf 540 6.0e-7, 5.1e-7 and 5.2e-7.
//
// Bound: FP32 issue, with the totals at two blocks an SM.  A point meets 54 (warp, group) sets of
// cells at width 9 (RPW = 4), 42 % of whose multiply-adds fall inside its support.  2e6 points in
// FP32, ms, the general kernel (integer shared-memory atomics) -> here: 8 channels 20.1 -> 6.32, 10
// channels 28.4 -> 7.61 (one word a sum and three blocks an SM: 4.80 and 6.05, at the price above).
// Folds every 16, 32, 64 steps: 6.56, 6.32, 6.20.  Float64, 2e4 points, 7 channels: 2.31 -> 1.71.
#include <algorithm>
#include <type_traits>

#include "fft_mixed.h"
#include "kernels.h"

namespace gpn {

namespace {

constexpr int kStrip = 8;                  // columns per lane group
constexpr int kGroups = 4;                 // lane groups per warp
constexpr int kTX = kStrip * kGroups;      // tile columns
constexpr int kTZ = 4;                     // tile planes
constexpr int kBands = 2;                  // row bands a plane
constexpr int kWarps = kTZ * kBands;
constexpr int kThreads = 32 * kWarps;
constexpr int kLists = kWarps * kGroups;
constexpr int kSlots = kThreads;           // points a batch (one a thread fills its tables)
constexpr int kScan = 4;                   // candidates a thread tests at a time
constexpr int kQueue = (kScan + 1) * kSlots;   // a scan adds up to kScan kSlots to less than kSlots
constexpr int kFold = 32;                  // list steps between folds into the totals (FP32)
constexpr int kMaxRanges = 64;             // bin rows a tile's candidates can come from

// per-slot shared tables (odd strides against bank conflicts); the row table has RPW - 1 zeros
// on either side, so a band row just outside the support reads zero without a test
__host__ __device__ constexpr int axis_stride(int w) { return w | 1; }
__host__ __device__ constexpr int row_stride(int w, int rpw) { return (w + 2 * (rpw - 1)) | 1; }
template <typename T>
__host__ __device__ constexpr int wk_pitch(int nc) {
  return (nc + (int)(16 / sizeof(T)) - 1) / (int)(16 / sizeof(T)) * (int)(16 / sizeof(T));
}

template <typename T>
struct Spread3Args {
  const int* l0[3];      // first support cell per axis (sorted order)
  const T* xi[3];
  const T* wk;           // [n][C]
  const int* bin_start;
  const int* tiles;      // active tile ids, (tz nty + ty) ntx + tx
  int ntx, nty;
  int nb[3];             // bins per axis
  int bt;                // bin edge in cells
  const double* alpha;   // sorted order, n x R column-major
  long long n;
  T* grid;
  GridView v;
  int width;
  T beta;
  T inv_halfw;
  int C;
};

// tot + acc <- tot + acc exactly: the rounded sum, and what it left out
__device__ __forceinline__ void fold(fft::f2& tot, fft::f2& acc) {
  const fft::f2 s = fft::vadd(tot, acc), b = fft::vsub(s, tot);
  acc = fft::vadd(fft::vsub(tot, fft::vsub(s, b)), fft::vsub(acc, b));
  tot = s;
}

// Blocks an SM.  A lane's sums take 8 RPW NC bytes (one float64 or two FP32 words each); of the
// registers left, 80 a thread do up to 160 bytes, 128 up to 320.
template <typename T, int NC, int RPW>
constexpr int kMinBlocks = 8 * RPW * NC <= 160 ? 3 : (8 * RPW * NC <= 320 || sizeof(T) == 8) ? 2 : 1;

// NC: channels held in registers (C itself up to 16, else 32 with the extra ones zero)
template <typename T, int NC, int RPW>
__global__ void __launch_bounds__(kThreads, (kMinBlocks<T, NC, RPW>)) k_spread3d(Spread3Args<T> a) {
  constexpr int TY = kBands * RPW, WP = wk_pitch<T>(NC), VW = (int)(16 / sizeof(T));
  // a sum: two channels (FP32) or one
  using Acc = typename std::conditional<sizeof(T) == 4, fft::f2, double>::type;
  constexpr int AL = fft::Elem<Acc>::lanes, NA = (NC + AL - 1) / AL;
  constexpr bool kTwo = AL == 2;   // totals apart from the running sums
  using V = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  const int W = a.width, PS = axis_stride(W), SY = row_stride(W, RPW), C = a.C, r = blockIdx.y;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* s_wk = reinterpret_cast<T*>(smem_raw);                      // [kSlots][WP]
  int4* s_l0 = reinterpret_cast<int4*>(s_wk + kSlots * WP);      // [kSlots]: (l0z, l0y, l0x, -)
  T* s_psx = reinterpret_cast<T*>(s_l0 + kSlots);                // [kSlots][PS]
  T* s_psz = s_psx + kSlots * PS;                                // [kSlots][PS]
  T* s_psy = s_psz + kSlots * PS;                                // [kSlots][SY]
  int* s_idx = reinterpret_cast<int*>(s_psy + kSlots * SY);      // [kQueue]: queue of points
  unsigned char* s_list = reinterpret_cast<unsigned char*>(s_idx + kQueue);      // [kLists][kSlots]
  __shared__ int s_rs[kMaxRanges], s_rl[kMaxRanges], s_wcnt[kScan][kWarps];
  __shared__ int s_cnt[kLists][kWarps], s_len[kLists];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = a.tiles[blockIdx.x], trow = tile / a.ntx;
  const int x0 = a.v.lo[2] + (tile - trow * a.ntx) * kTX;
  const int y0 = a.v.lo[1] + (trow % a.nty) * TY, z0 = a.v.lo[0] + trow / a.nty * kTZ;

  // candidates: per bin row one contiguous run of sorted points
  auto first_bin = [&](int c0) { return max(0, c0 - W + 1) / a.bt; };
  const int bz0 = first_bin(z0), nz = min(a.nb[0] - 1, (z0 + kTZ - 1) / a.bt) - bz0 + 1;
  const int by0 = first_bin(y0), ny = min(a.nb[1] - 1, (y0 + TY - 1) / a.bt) - by0 + 1;
  const int bx0 = first_bin(x0), bx1 = min(a.nb[2] - 1, (x0 + kTX - 1) / a.bt);
  const int nr = min(kMaxRanges, max(nz, 0) * max(ny, 0));
  if (tid < nr) {
    const int qz = tid / ny, qy = tid - qz * ny;
    const long long row = ((long long)(bz0 + qz) * a.nb[1] + by0 + qy) * a.nb[2];
    const int lo = a.bin_start[row + bx0];
    s_rs[tid] = lo;
    s_rl[tid] = a.bin_start[row + bx1 + 1] - lo;
  }
  __syncthreads();
  int total = 0;
  for (int q = 0; q < nr; ++q) total += s_rl[q];

  Acc acc[RPW][NA], tot[kTwo ? RPW : 1][kTwo ? NA : 1];
#pragma unroll
  for (int rr = 0; rr < RPW; ++rr)
#pragma unroll
    for (int k = 0; k < NA; ++k) {
      acc[rr][k] = fft::vset<Acc>(T(0));
      if constexpr (kTwo) tot[rr][k] = fft::vset<Acc>(T(0));
    }
  const int grp = lane >> 3;
  const int xg = x0 + grp * kStrip + (lane & 7);                     // this lane's column
  const int zw = z0 + warp / kBands, rw0 = y0 + warp % kBands * RPW;  // the warp's plane, first row
  const int my_list = warp * kGroups + grp;
  const unsigned lt = (1u << lane) - 1u;
  const double* alpha_r = a.alpha + (size_t)r * a.n;

  int queued = 0;
  for (int c0 = 0; c0 < total || queued > 0; ) {
    if (c0 < total && queued < kSlots) {
      // scan: kScan candidates per thread (their cells are loaded before the first test); the
      // ones meeting the tile join the queue in order
      int p[kScan];
      unsigned bal[kScan];
      bool meets[kScan];
#pragma unroll
      for (int i = 0; i < kScan; ++i) {
        int c = c0 + i * kThreads + tid;
        meets[i] = c < total;
        p[i] = 0;
        if (meets[i]) {
          for (int q = 0; q < nr; ++q) {
            if (c < s_rl[q]) {
              p[i] = s_rs[q] + c;
              break;
            }
            c -= s_rl[q];
          }
        }
      }
      int lz[kScan], ly[kScan], lx[kScan];
#pragma unroll
      for (int i = 0; i < kScan; ++i) {
        lz[i] = a.l0[0][p[i]];
        ly[i] = a.l0[1][p[i]];
        lx[i] = a.l0[2][p[i]];
      }
#pragma unroll
      for (int i = 0; i < kScan; ++i) {
        meets[i] = meets[i] && lz[i] + W > z0 && lz[i] < z0 + kTZ && ly[i] + W > y0 && ly[i] < y0 + TY &&
                   lx[i] + W > x0 && lx[i] < x0 + kTX;
        bal[i] = __ballot_sync(0xffffffffu, meets[i]);
        if (lane == 0) s_wcnt[i][warp] = __popc(bal[i]);
      }
      __syncthreads();
      int end = queued;
#pragma unroll
      for (int i = 0; i < kScan; ++i) {
        int off = end;
#pragma unroll
        for (int q = 0; q < kWarps; ++q) {
          const int v = s_wcnt[i][q];
          off += q < warp ? v : 0;
          end += v;
        }
        if (meets[i]) s_idx[off + __popc(bal[i] & lt)] = p[i];
      }
      queued = end;
      c0 += kScan * kThreads;
      __syncthreads();
      if (queued < kSlots && c0 < total) continue;
    }
    // a batch: tables of its points, one per thread
    const int nb = min(queued, kSlots);
    unsigned mask = 0u;   // the (warp, group) lists the support meets
    if (tid < nb) {
      const int p = s_idx[tid];
      const int lz = a.l0[0][p], ly = a.l0[1][p], lx = a.l0[2][p];
      const int b0 = ly <= y0 ? 0 : (ly - y0) / RPW, b1 = min(kBands - 1, (ly + W - 1 - y0) / RPW);
      const int s0 = lx <= x0 ? 0 : (lx - x0) / kStrip, s1 = min(kGroups - 1, (lx + W - 1 - x0) / kStrip);
      const unsigned smask = ((1u << (s1 + 1)) - 1u) & ~((1u << s0) - 1u);
      unsigned bands = 0u;
      for (int b = b0; b <= b1; ++b) bands |= smask << (b * kGroups);
      const int q0 = max(0, lz - z0), q1 = min(kTZ - 1, lz + W - 1 - z0);
      for (int q = q0; q <= q1; ++q) mask |= bands << (q * kBands * kGroups);
      s_l0[tid] = make_int4(lz, ly, lx, 0);
      const T zq = a.xi[0][p], yq = a.xi[1][p], xq = a.xi[2][p];
      T* px = s_psx + tid * PS;
      T* pz = s_psz + tid * PS;
      T* py = s_psy + tid * SY;
      for (int j = 0; j < W; ++j) {
        px[j] = psi_at<T>(j, xq, a.beta, a.inv_halfw);
        pz[j] = psi_at<T>(j, zq, a.beta, a.inv_halfw);
      }
      for (int j = 0; j < SY; ++j) {
        const int jj = j - (RPW - 1);
        py[j] = (jj >= 0 && jj < W) ? psi_at<T>(jj, yq, a.beta, a.inv_halfw) : T(0);
      }
      const T amp = (T)alpha_r[p];
      const T* wkp = a.wk + (size_t)p * C;
#pragma unroll
      for (int k = 0; k < WP; ++k) s_wk[tid * WP + k] = k < C ? wkp[k] * amp : T(0);
    }
#pragma unroll
    for (int L = 0; L < kLists; ++L) {
      const unsigned bl = __ballot_sync(0xffffffffu, (mask >> L) & 1u);
      if (lane == 0) s_cnt[L][warp] = __popc(bl);
    }
    __syncthreads();
    // exclusive prefix over warps of every list count: warp w scans lists 4w .. 4w + 3
    {
      const int L = warp * kGroups + (lane >> 3), q = lane & 7;
      const int v = s_cnt[L][q];
      int inc = v;
#pragma unroll
      for (int o = 1; o < 8; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, o, 8);
        if (q >= o) inc += u;
      }
      __syncwarp();
      s_cnt[L][q] = inc - v;
      if (q == 7) s_len[L] = inc;
    }
    // the queue's rest moves to its front
    const int rest = queued - nb;
    int moved[kScan];
#pragma unroll
    for (int i = 0; i < kScan; ++i) moved[i] = i * kThreads + tid < rest ? s_idx[kSlots + i * kThreads + tid] : 0;
    __syncthreads();
#pragma unroll
    for (int i = 0; i < kScan; ++i)
      if (i * kThreads + tid < rest) s_idx[i * kThreads + tid] = moved[i];
    queued = rest;
#pragma unroll
    for (int L = 0; L < kLists; ++L) {
      const unsigned hit = (mask >> L) & 1u;
      const unsigned bl = __ballot_sync(0xffffffffu, hit);
      if (hit) s_list[L * kSlots + s_cnt[L][warp] + __popc(bl & lt)] = (unsigned char)tid;
    }
    __syncthreads();
    // accumulate: group g walks the list of (its warp, strip g)
    const int len = s_len[my_list];
    int steps = 0;
#pragma unroll
    for (int q = 0; q < kGroups; ++q) steps = max(steps, s_len[warp * kGroups + q]);
    const unsigned char* lst = s_list + my_list * kSlots;
    for (int j0 = 0; j0 < steps; j0 += kFold) {
      const int j1 = min(j0 + kFold, steps);
      for (int j = j0; j < j1; ++j) {
        const bool ok = j < len;
        const int is = ok ? lst[j] : 0;
        const int4 l0 = s_l0[is];
        const int dx = xg - l0.z;
        const bool in = ok && (unsigned)dx < (unsigned)W;
        const T pxz = in ? s_psx[is * PS + dx] * s_psz[is * PS + (zw - l0.x)] : T(0);
        Acc wk[WP / AL];
#pragma unroll
        for (int v = 0; v < WP / VW; ++v) {
          const V u = reinterpret_cast<const V*>(s_wk + is * WP)[v];
          if constexpr (VW == 4) {
            wk[2 * v] = {u.x, u.y};
            wk[2 * v + 1] = {u.z, u.w};
          } else {
            wk[2 * v] = u.x;
            wk[2 * v + 1] = u.y;
          }
        }
        // rows of the band relative to the support: in [1 - RPW, W - 1] for list members
        const T* pyr = s_psy + is * SY + (RPW - 1) + (ok ? rw0 - l0.y : 0);
#pragma unroll
        for (int rr = 0; rr < RPW; ++rr) {
          const Acc v = fft::vset<Acc>(pxz * pyr[rr]);
#pragma unroll
          for (int k = 0; k < NA; ++k) acc[rr][k] = fft::vfma(v, wk[k], acc[rr][k]);
        }
      }
      if constexpr (kTwo) {
#pragma unroll
        for (int rr = 0; rr < RPW; ++rr)
#pragma unroll
          for (int k = 0; k < NA; ++k) fold(tot[rr][k], acc[rr][k]);
      }
    }
    __syncthreads();  // slots, lists and counters are refilled by the next batch
  }

  // every lane holds the complete sums of its column over the warp's rows
  const int gx = xg - a.v.lo[2], gz = zw - a.v.lo[0];
  if (gx >= a.v.ext[2] || gz >= a.v.ext[0]) return;
  T* gr = a.grid + r * a.v.rstride + gz * a.v.stride[0] + gx * a.v.stride[2];
#pragma unroll
  for (int rr = 0; rr < RPW; ++rr) {
    const int gy = rw0 + rr - a.v.lo[1];
    if (gy < a.v.ext[1]) {
      T* o = gr + gy * a.v.stride[1];
      // whole sums: the pitch holds them (in FP32 it is even, a padding channel's weights are zero)
#pragma unroll
      for (int k = 0; k < NA; ++k)
        if (k * AL < C) {
          if constexpr (kTwo) acc[rr][k] = fft::vadd(tot[rr][k], acc[rr][k]);
          *reinterpret_cast<Acc*>(o + k * AL) = acc[rr][k];
        }
    }
  }
}

constexpr int reg_channels(int C) { return C <= 16 ? C : 32; }
// four rows a warp up to the channels whose sums leave two blocks an SM (12 channels, 5e5 points at
// width 8: 1.66 ms with two rows, 2.09 with four and one block; 8 and 10 channels above: 6.58 and
// 9.00 ms with two)
template <typename T>
constexpr int rows_per_warp(int nc) { return (sizeof(T) == 8 || nc > 10) ? 2 : 4; }

size_t smem_bytes(size_t rs, int nc, int rpw, int w) {
  const int wp = rs == 4 ? wk_pitch<float>(nc) : wk_pitch<double>(nc);
  return (size_t)kSlots * ((2 * axis_stride(w) + row_stride(w, rpw) + wp) * rs + sizeof(int4) + kLists) +
         sizeof(int) * kQueue;
}

template <typename T, int NC>
void launch(const Spread3Args<T>& a, dim3 grid, cudaStream_t st) {
  constexpr int RPW = rows_per_warp<T>(NC);
  const size_t smem = smem_bytes(sizeof(T), NC, RPW, a.width);
  GPN_CUDA(cudaFuncSetAttribute(k_spread3d<T, NC, RPW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  k_spread3d<T, NC, RPW><<<grid, kThreads, smem, st>>>(a);
}

template <typename T, int NC>
void dispatch(const Spread3Args<T>& a, dim3 grid, cudaStream_t st) {
  if constexpr (NC > 16) {
    launch<T, 32>(a, grid, st);
  } else {
    if (a.C == NC)
      launch<T, NC>(a, grid, st);
    else
      dispatch<T, NC + 1>(a, grid, st);
  }
}

template <typename T>
void impl(Plan& plan, const double* alpha_sorted, int R, cudaStream_t st) {
  if (plan.n_sp3_tiles == 0) return;
  const GridGeom& g = plan.geom;
  const PointSet& ps = plan.pts;
  Spread3Args<T> a{};
  for (int q = 0; q < 3; ++q) {
    a.l0[q] = ps.cell0[q];
    a.xi[q] = (const T*)ps.xi[q];
    a.nb[q] = ps.nbins[q];
  }
  a.wk = (const T*)ps.wk;
  a.bin_start = ps.bin_start;
  a.tiles = plan.sp3_tiles;
  a.v = plan.view;
  const int TY = kBands * rows_per_warp<T>(reg_channels(g.C));
  a.ntx = (a.v.ext[2] + kTX - 1) / kTX;
  a.nty = (a.v.ext[1] + TY - 1) / TY;
  a.bt = g.tile;
  a.alpha = alpha_sorted;
  a.n = ps.n;
  a.grid = (T*)plan.grid;
  a.width = g.width;
  a.beta = es_beta_arg<T>(g.beta);
  a.inv_halfw = (T)(2.0 / g.width);
  a.C = g.C;
  dispatch<T, 1>(a, dim3((unsigned)plan.n_sp3_tiles, (unsigned)R), st);
  GPN_CUDA(cudaGetLastError());
}

int tile_rows(const Plan& plan) {
  const int nc = reg_channels(plan.geom.C);
  return kBands * (plan.precision == GP_FP32 ? rows_per_warp<float>(nc) : rows_per_warp<double>(nc));
}

}  // namespace

// Tiles whose candidate bins hold at least one point; the others stay zero.
void build_spread3d_tiles(Plan& plan, const std::vector<int>& bstart) {
  const GridGeom& g = plan.geom;
  const PointSet& ps = plan.pts;
  const GridView& v = plan.view;
  const int TY = tile_rows(plan), edge[3] = {kTZ, TY, kTX};
  // the candidate table and the shared memory hold every box plan (bins are at least a support
  // less a cell wide: at most 16 bin rows, and 191488 bytes with 32 float64 channels at width 16)
  const int rows = ((kTZ + g.width - 2) / g.tile + 2) * ((TY + g.width - 2) / g.tile + 2);
  GPN_CHECK(rows <= kMaxRanges && smem_bytes(plan.real_size, reg_channels(g.C), TY / kBands, g.width) <= 200 * 1024,
            GP_EUNSUPPORTED, "3-D spread: bins too narrow or too many channels");
  int nt[3];
  std::vector<int> lo[3], hi[3];   // bins a tile's candidates come from, per axis
  for (int q = 0; q < 3; ++q) {
    nt[q] = (v.ext[q] + edge[q] - 1) / edge[q];
    for (int t = 0; t < nt[q]; ++t) {
      const int c0 = v.lo[q] + t * edge[q];
      lo[q].push_back(std::max(0, c0 - g.width + 1) / g.tile);
      hi[q].push_back(std::min(ps.nbins[q] - 1, (c0 + edge[q] - 1) / g.tile));
    }
  }
  GPN_CHECK((long long)nt[0] * nt[1] * nt[2] < (1ll << 31), GP_EINVAL, "too many tiles");
  std::vector<int> act;
  for (int tz = 0; tz < nt[0]; ++tz)
    for (int ty = 0; ty < nt[1]; ++ty)
      for (int tx = 0; tx < nt[2]; ++tx) {
        bool any = false;
        for (int bz = lo[0][tz]; bz <= hi[0][tz] && !any; ++bz)
          for (int by = lo[1][ty]; by <= hi[1][ty] && !any; ++by) {
            const size_t row = ((size_t)bz * ps.nbins[1] + by) * ps.nbins[2];
            any = bstart[row + hi[2][tx] + 1] > bstart[row + lo[2][tx]];
          }
        if (any) act.push_back((tz * nt[1] + ty) * nt[2] + tx);
      }
  plan.n_sp3_tiles = (long long)act.size();
  plan.sp3_tiles = (int*)plan.alloc(sizeof(int) * std::max<size_t>(act.size(), 1));
  if (!act.empty())
    GPN_CUDA(cudaMemcpy(plan.sp3_tiles, act.data(), sizeof(int) * act.size(), cudaMemcpyHostToDevice));
}

void launch_spread3d(Plan& plan, const double* alpha_sorted, int R, cudaStream_t st) {
  if (plan.precision == GP_FP32)
    impl<float>(plan, alpha_sorted, R, st);
  else
    impl<double>(plan, alpha_sorted, R, st);
}

}  // namespace gpn
