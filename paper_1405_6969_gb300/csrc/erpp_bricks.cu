// erpp_bricks.cu -- particles sorted by 8 x 8 x 8-cell bricks, and the FP32
// regularised source from them (Sec. 2.4, Eq. ns_regularized_filtered) as a
// tensor-core contraction.
//
// Bricks.  A particle belongs to the brick of its home cell and is recorded
// once (the x/y-halo tiles cut a stencil into pieces and record each).  Bricks
// are numbered group by group of 2 x 2 x 2, so that the 16 x 16 x 16 cells of a
// group, and the 16 x 16 x 8 of half of one, are one range of records.  The
// sort is a counting sort by brick (k_brick_count, a scan, k_brick_place)
// followed by k_brick_order, which puts the members of a brick in index
// order: the order of the records, and with it every sum taken over them,
// does not depend on the order in which the counting atomics arrived (bricks
// of more than kOrderMax members keep the order of arrival).
//
// Source.  S_c(z, y, x) = sum_p (e_z e_y)(z, y; p) (f_c e_x)(x; p) over the
// particles whose windows reach the region: a matrix product with the
// particles as its inner dimension.  A block owns a region of 16 x 16 x 16
// nodes; it lists the particles that touch it from the bricks around, and for
// every batch of the list stages per particle the y- and z-weights (FP32) and
// the products f_c e_x of the 16 columns.  Each of the 16 warps owns two
// planes of eight rows, and accumulates 16 particles at a time in registers
// with mma.m16n8k16 (rows: 2 planes x 8 rows; columns: 8 nodes of x; inner
// dimension: the particles that reach the warp's rows, compacted).  Nothing is
// added by atomics, the region needs no halo, and S is written once.
//
// Precision.  Both factors are split into two FP16 numbers, v = h + l (h the
// rounded value, l the rounded rest: off by at most 2^-23 |v|, 2^-24.5 rms), and the
// three products h h', h l', l h' are summed in FP32, 16 particles at a time; the
// chunks' sums are added in FP32 with rounding (the tensor core truncates:
// accumulating through it, 125 chunks of a dense cluster left an error of 1.5e-5).
// The dropped l l' is at most 2^-22 of its term (|l| <= 2^-11 |v|), 2^-24.6 rms.  The
// factors are scaled by powers of two so that a term of 2^-17 of the largest is
// still split without underflow; a smaller one keeps an error of 2^-39 of the largest
// (a tile's fixed point: 2^-31 of the sum of its forces).  Against 64 bits, S is at
// most as far off as from the tiles, relative to the whole and to each node's own
// terms: 100k particles in clusters 2.0e-7 of the whole and 4.8e-8 of a node's in the
// median, tiles 1.5e-6 and 1.2e-7; 800k uniform ones 1.9e-7 and 3.6e-8, tiles 2.2e-7
// and 4.1e-8; the same with forces spread over nine decades.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdlib.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "erpp_internal.cuh"

namespace {

constexpr int kOrderMax = 4096;  // members of a brick put in index order, at most

__device__ __forceinline__ int brick_id(const int ng[3], int bx, int by, int bz) {
  const int g = ((bz >> 1) * ng[1] + (by >> 1)) * ng[0] + (bx >> 1);
  return g * 8 + ((bz & 1) << 2) + ((by & 1) << 1) + (bx & 1);
}

// Window, home cell and brick of every particle; its place among the members
// of the brick by order of arrival.  Invalid positions get brick -1.
__global__ void __launch_bounds__(256) k_brick_count(erpp_kparams kp, erpp_brick_dims bd,
                                                     int64_t n, const double* __restrict__ x0,
                                                     const double* __restrict__ x1,
                                                     const double* __restrict__ x2,
                                                     float4* __restrict__ rec_in,
                                                     int2* __restrict__ key,
                                                     int32_t* __restrict__ cnt, uint32_t* err) {
  erpp_pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double xv[3] = {x0[i], x1[i], x2[i]};
  bool ok = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // 0 <= x < L on the bit patterns (-0 is in range, NaN is not)
    const unsigned long long bits = (unsigned long long)__double_as_longlong(xv[a]);
    ok = ok && (bits < (unsigned long long)__double_as_longlong(kp.L[a]) || (bits << 1) == 0ull);
  }
  if (!ok) {
    erpp_set_err(err, ERPP_ERRBIT_RANGE);
    key[i] = make_int2(-1, 0);
    return;
  }
  int c[3];
  float t[3];
  uint32_t w = 0;
  bool inb = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const erpp_axis_win aw =
        erpp_axis_window_lean(xv[a], kp.inv_dx[a], kp.cp[a], kp.cp_int[a], kp.cp_frac[a]);
    const int off = aw.lo - aw.ci, nw = aw.hi - aw.lo + 1;
    inb = inb && off >= -kp.hlo && off <= 0 && nw >= 1 && nw <= kp.xs;
    // s can round up to exactly N: the first cell of the next image
    c[a] = aw.ci >= kp.n[a] ? aw.ci - kp.n[a] : aw.ci;
    t[a] = aw.t;
    // off is -ck - 1, -ck or -ck + 1 (ck = floor(c'), the first by rounding)
    const int so = off + kp.cp_int[a] + 1;
    inb = inb && so >= 0 && so <= 3;
    w |= (uint32_t)((c[a] & 7) + off + 8) << (8 * a) | (uint32_t)nw << (8 * a + 4) |
         (uint32_t)so << (24 + 2 * a);
  }
  if (!inb) {
    erpp_set_err(err, ERPP_ERRBIT_BOUNDS);
    key[i] = make_int2(-1, 0);
    return;
  }
  const int b = brick_id(bd.ng, c[0] >> 3, c[1] >> 3, c[2] >> 3);
  rec_in[i] = make_float4(t[0], t[1], t[2], __uint_as_float(w));
  key[i] = make_int2(b, atomicAdd(&cnt[b], 1));
}

// Exclusive scan of the brick counts in one launch, 4096 counts a block: each
// block also adds up all the counts before its own (2 MB of L2 reads in all for
// 65536 bricks), so that no block waits for another.  Up to kBrickScanOne
// bricks; beyond, where those reads grow, the three-kernel scan.
constexpr int kBrickScanOne = 131072;
__global__ void __launch_bounds__(1024) k_brick_scan(const int32_t* __restrict__ cnt,
                                                     int32_t* __restrict__ start, int nb) {
  __shared__ int32_t ws[32], wp[32];
  erpp_pdl_enter();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int base = blockIdx.x * 4096;
  int32_t before = 0;
#pragma unroll 8
  for (int k = threadIdx.x * 4; k < base; k += 4096) {
    const int4 v = *reinterpret_cast<const int4*>(cnt + k);
    before += v.x + v.y + v.z + v.w;
  }
  const int at = base + threadIdx.x * 4;  // nb is a multiple of 8
  const int4 v = at < nb ? *reinterpret_cast<const int4*>(cnt + at) : make_int4(0, 0, 0, 0);
  const int32_t s = v.x + v.y + v.z + v.w;
  int32_t incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
    before += __shfl_xor_sync(0xffffffffu, before, o);
  }
  if (lane == 31) ws[warp] = incl;
  if (lane == 0) wp[warp] = before;
  __syncthreads();
  int32_t wi = ws[lane], all = wp[lane];
  const int32_t own = wi;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t u = __shfl_up_sync(0xffffffffu, wi, o);
    if (lane >= o) wi += u;
    all += __shfl_xor_sync(0xffffffffu, all, o);
  }
  const int32_t pre = __shfl_sync(0xffffffffu, wi - own, warp);
  const int32_t tot = __shfl_sync(0xffffffffu, wi, 31);
  if (at < nb) {
    int4 o;
    o.x = all + pre + incl - s;
    o.y = o.x + v.x;
    o.z = o.y + v.y;
    o.w = o.z + v.z;
    *reinterpret_cast<int4*>(start + at) = o;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) start[nb] = all + tot;
}

// Records of the adjoint's particles: the particle of each, and the further chunks
// of tiles of more than `chunk` particles.
struct AdjOrder {
  int32_t* ord;  // null: not for the adjoint
  int32_t* nitems;
  int2* items;
  int tile_bricks, chunk;
  __device__ __forceinline__ void put(int pos, int i, int brick,
                                      const int32_t* __restrict__ start) const {
    ord[pos] = i;
    const int tile = brick / tile_bricks;
    const int off = pos - start[tile * tile_bricks];
    if (off >= chunk && off % chunk == 0) items[atomicAdd(nitems, 1)] = make_int2(tile, pos);
  }
};

// adj.ord given: the records' final places, in order of arrival.  An adjoint alone
// takes them so: each particle's sums are its own, whatever the order.
__global__ void __launch_bounds__(256) k_brick_place(int64_t n, const int2* __restrict__ key,
                                                     const float4* __restrict__ rec_in,
                                                     const int32_t* __restrict__ start,
                                                     float4* __restrict__ rec_tmp,
                                                     int32_t* __restrict__ pidx,
                                                     int32_t* __restrict__ pbrick,
                                                     int32_t* __restrict__ slot, AdjOrder adj) {
  erpp_pdl_enter();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int2 k = key[i];
  if (k.x < 0) {
    slot[i] = -1;
    return;
  }
  const int pos = start[k.x] + k.y;
  rec_tmp[pos] = rec_in[i];
  if (adj.ord) {
    slot[i] = pos;
    adj.put(pos, (int)i, k.x, start);
    return;
  }
  pidx[pos] = (int)i;
  pbrick[pos] = k.x;
}

// A brick is dense that holds this many particles and more than an eighth of an
// SM's share of all n: its regions take so long that the others are done before.
// Uniform clouds of about 200 per brick, one source by whole regions and by
// quarters: 64^3 292 and 198 us, 72^3 343 and 295, 80^3 356 and 341; where every
// SM has its regions anyway 96^3 378 and 485, 128^3 565 and 848 us.
constexpr int kDenseBrick = 192;
static_assert(kDenseBrick >= 64, "mark_dense's members");
__device__ __forceinline__ bool dense_brick(int members, int64_t n) {
  return members >= kDenseBrick && members > n / (8 * ERPP_SMS);
}
// Lists the regions that the members of a dense brick can reach, each once: the r-th
// of its first 64 members the r-th of up to 4 x 4 x 4 (one member listed them all, one
// atomic after the other, while the rest of the sort had long been done: 10.5k
// particles in 50 clusters, k_brick_order 21.5 us, now 8.8).
// Called instead of inlined it cost the ranking's registers: 400k particles in clusters
// 112 us instead of 84.
__device__ __forceinline__ void mark_dense(const erpp_kparams& kp, const erpp_brick_dims& bd,
                                           int id, int r, int32_t* ndense, int32_t* dense,
                                           int32_t* dflag) {
  int g = id >> 3;
  const int br[3] = {2 * (g % bd.ng[0]) + (id & 1), 2 * ((g / bd.ng[0]) % bd.ng[1]) + ((id >> 1) & 1),
                     2 * (g / (bd.ng[0] * bd.ng[1])) + ((id >> 2) & 1)};
  int at[3];
  for (int a = 0; a < 3; ++a) {
    // the want-th region along the axis, from the lowest node that is reached
    const int n = kp.n[a], last = min(8 * br[a] + 8, n) + kp.hlo, want = (r >> (2 * a)) & 3;
    int k = 0, j = 8 * br[a] - kp.hlo;
    for (; j <= last; ++k) {
      const int w = j - erpp_floordiv(j, n) * n;
      if (k == want) {
        at[a] = w >> 4;
        break;
      }
      j += min(((w >> 4) + 1) * 16, n) - w;
    }
    if (j > last) return;  // fewer regions than that
  }
  g = (at[2] * bd.ng[1] + at[1]) * bd.ng[0] + at[0];
  if (atomicExch(&dflag[g], 1) == 0) dense[atomicAdd(ndense, 1)] = g;
}

// Position j's particle moves to its rank (by index) among its brick's members.
// The threads of a warp mostly share a brick, so its indices are read as
// broadcasts, 16 bytes at a time (a dense cluster's bricks hold a thousand
// members: 95 us one index at a time for 100k particles in such bricks).
__global__ void __launch_bounds__(256) k_brick_order(int64_t n, int nb,
                                                     const int32_t* __restrict__ pidx,
                                                     const int32_t* __restrict__ pbrick,
                                                     const float4* __restrict__ rec_tmp,
                                                     const int32_t* __restrict__ start,
                                                     float4* __restrict__ rec,
                                                     uint32_t* __restrict__ win,
                                                     int32_t* __restrict__ slot, AdjOrder adj,
                                                     erpp_kparams kp, erpp_brick_dims bd,
                                                     int32_t* __restrict__ ndense,
                                                     int32_t* __restrict__ dense,
                                                     int32_t* __restrict__ dflag) {
  erpp_pdl_enter();
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n || j >= start[nb]) return;
  const int me = pidx[j], b = pbrick[j];
  const float4 v = rec_tmp[j];
  const int s = start[b], e = start[b + 1];
  int r = 0;
  if (e - s <= kOrderMax) {
    int k = s;
    const int body = min((s + 3) & ~3, e), tail = max(e & ~3, body);
    for (; k < body; ++k) r += pidx[k] < me ? 1 : 0;
#pragma unroll 4
    for (; k < tail; k += 4) {
      const int4 q = *reinterpret_cast<const int4*>(pidx + k);
      r += (q.x < me ? 1 : 0) + (q.y < me ? 1 : 0) + (q.z < me ? 1 : 0) + (q.w < me ? 1 : 0);
    }
    for (; k < e; ++k) r += pidx[k] < me ? 1 : 0;
  } else {
    r = (int)j - s;
  }
  rec[s + r] = v;
  win[s + r] = __float_as_uint(v.w);
  slot[me] = s + r;
  if (r < 64 && dense_brick(e - s, n)) mark_dense(kp, bd, b, r, ndense, dense, dflag);
  if (adj.ord) adj.put(s + r, me, b, start);
}

// Normalisation of a particle's weights (erpp_norm's arithmetic on its record).
__device__ __forceinline__ float rec_norm(const erpp_kparams& kp, float4 r) {
  if (!kp.normalize) return (float)(kp.dV * kp.raw_norm3);
  const uint32_t w = __float_as_uint(r.w);
  const float t[3] = {r.x, r.y, r.z};
  float prod = 1.f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int nw = erpp_rec_nw(w, a), off = erpp_rec_off(kp, w, a);
    float sum = 0.f;
    for (int k = 0; k < nw; ++k) {
      const float d = (float)(off + k) - t[a];
      sum += erpp_ex2(-kp.beta[a] * d * d);
    }
    prod *= sum;
  }
  return 1.f / prod;
}

__global__ void __launch_bounds__(256) k_brick_forces(erpp_kparams kp, int64_t n,
                                                      const double* __restrict__ D0,
                                                      const double* __restrict__ D1,
                                                      const double* __restrict__ D2, float scale,
                                                      const float4* __restrict__ rec,
                                                      const int2* __restrict__ key,
                                                      const int32_t* __restrict__ slot,
                                                      float4* __restrict__ fs,
                                                      int32_t* __restrict__ bmax) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int sl = slot[i];
  if (sl < 0) return;
  const float s = rec_norm(kp, rec[sl]) * scale;
  erpp_put_force(fs, bmax, sl, key[i].x, s * (float)D0[i], s * (float)D1[i], s * (float)D2[i]);
}

// ---- the source ----
constexpr int kRegion = 16;      // nodes of a region per axis
constexpr int kListBatch = 296;  // particles staged at a time, at most
constexpr int kScatThreads = 512;
constexpr int kScatWarps = kScatThreads / 32;
// A warp's own list area: offsets of the rows it works on, from its start; the
// queue of the members that it found, 4 bytes each, from its end.
constexpr int kArea = 896;
constexpr int kQueueMost = 4096;  // members of a segment whose places an entry can hold
// Staged row of a particle: 3 components x (h, l) x 16 columns of FP16, 16 y-
// and 16 z-weights (FP32).  The pitch puts the rows that an ldmatrix (eight consecutive particles) or a
// fragment load (four, every other one) reads together in different banks.
constexpr int kRowW = 192;
constexpr int kPitch = 336;
constexpr int kMaxAxisSegs = 8;  // at most 6 are used
constexpr int kMaxSegs = 352;

__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// The same with a zero addend.
__device__ __forceinline__ void mma_f16_zero(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                             uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%10,%10,%10,%10};\n"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
// A pair of FP32 values in one register pair: one instruction works on both,
// each rounded as by itself.
struct Pair {
  unsigned long long v;
};
__device__ __forceinline__ Pair pair_of(float a, float b) {
  Pair p;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(p.v) : "f"(a), "f"(b));
  return p;
}
__device__ __forceinline__ float2 parts(Pair p) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;\n" : "=f"(f.x), "=f"(f.y) : "l"(p.v));
  return f;
}
__device__ __forceinline__ Pair operator+(Pair a, Pair b) {
  Pair p;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(p.v) : "l"(a.v), "l"(b.v));
  return p;
}
__device__ __forceinline__ Pair operator*(Pair a, Pair b) {
  Pair p;
  asm("mul.rn.f32x2 %0, %1, %2;\n" : "=l"(p.v) : "l"(a.v), "l"(b.v));
  return p;
}
// v = h + l in FP16 for a pair of values.
__device__ __forceinline__ void split_pair(Pair v, uint32_t& h, uint32_t& l) {
  const float2 f = parts(v);
  const __half2 hh = __floats2half2_rn(f.x, f.y);
  const float2 hf = __half22float2(hh);
  const float2 rest = parts(v + pair_of(-hf.x, -hf.y));
  const __half2 ll = __floats2half2_rn(rest.x, rest.y);
  h = *reinterpret_cast<const uint32_t*>(&hh);
  l = *reinterpret_cast<const uint32_t*>(&ll);
}

struct ScatShared {
  int cnt[kScatWarps];  // members each warp found that touch the region
  int maxbits;          // largest |force component| of the bricks around
  int odd;              // a staged particle's force is not finite
};

// Dense regions: the segments one after the other as one range of candidates,
// and how many of the candidates before every G-th touch the region.  In the
// last rows' place (dense batches are shorter).
constexpr int kDenseBatch = 272;
constexpr int kMarks = 512;
struct DenseTab {
  int start[kMaxSegs];   // first record of the segment's brick, less the candidates before
  uint32_t org[kMaxSegs];
  int pre[kMaxSegs + 1]; // candidates before the segment
  int mark[kMarks + 1];
};
static_assert(sizeof(DenseTab) <= (kListBatch - kDenseBatch) * kPitch, "dense table");

// Largest k in [0, n) with v[k] <= x (v ascending, v[0] <= x).
__device__ __forceinline__ int last_not_above(const int* v, int n, int x) {
  int lo = 0, hi = n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (v[mid] <= x) lo = mid; else hi = mid;
  }
  return lo;
}
// Exclusive scan of v[0..n) in place by one warp, total at v[n].
__device__ __forceinline__ void warp_scan(int* v, int n, int lane) {
  int carry = 0;
  for (int q0 = 0; q0 < n; q0 += 32) {
    const int x = q0 + lane < n ? v[q0 + lane] : 0;
    int incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += u;
    }
    if (q0 + lane < n) v[q0 + lane] = carry + incl - x;
    carry += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) v[n] = carry;
}

// A particle's window relative to a region, all axes at once in the bytes of
// a word: first node + 64.
__device__ __forceinline__ uint32_t window_lo(uint32_t w, uint32_t org) {
  return (w & 0x0f0f0fu) + org;
}
// Whether the window reaches nodes [0, ext) on every axis; ext1 holds 63 + ext
// per byte, with the top bits set: lo < ext leaves the top bit of ext1 - (lo +
// 64), and lo + length > 0 carries (lo + 64) + length + 63 into the top bit.
__device__ __forceinline__ bool touches(uint32_t w, uint32_t org, uint32_t ext1) {
  const uint32_t lo = window_lo(w, org);
  const uint32_t hi = lo + ((w >> 4) & 0x0f0f0fu) + 0x3f3f3fu;
  return (((ext1 - lo) & hi) & 0x808080u) == 0x808080u;
}

// A region of more than this many particles (a quarter of one, kOddQuarter) passes
// forces that are not finite on to the nodes in their windows; elsewhere such a
// component gives nothing.  The tiles do the same: a tile of 64 x 16 x 4 nodes sums
// up to 1024 pieces in fixed point, which has no such values, and more in FP32; a
// region and a tile of the same density hold as many, a quarter 0.43 times.
constexpr int kOddRegion = 1024, kOddQuarter = 440;

// Adds them, after S has its finite sums: the whole block, a thread per particle of
// the bricks around (seldom called, so that it keeps out of scatter_region's registers).
__device__ __noinline__ void add_odd_forces(const erpp_kparams& kp, const erpp_brick_dims& bd,
                                            const int gg0, const int gg1, const int gg2, int z0,
                                            int zs, const int2* __restrict__ axis,
                                            const uint32_t* __restrict__ win,
                                            const float4* __restrict__ fs,
                                            const int32_t* __restrict__ bstart, float* S) {
  const int b[3] = {gg0 * kRegion, gg1 * kRegion, gg2 * kRegion + z0};
  const int ext[3] = {min(kRegion, kp.n[0] - b[0]), min(kRegion, kp.n[1] - b[1]),
                      min(zs, kp.n[2] - b[2])};
  const int2* ax[3] = {axis + (size_t)gg0 * kMaxAxisSegs,
                       axis + (size_t)(bd.ng[0] + gg1) * kMaxAxisSegs,
                       axis + (size_t)(bd.ng[0] + bd.ng[1] + gg2) * kMaxAxisSegs};
  const int ns[3] = {ax[0][kMaxAxisSegs - 1].x, ax[1][kMaxAxisSegs - 1].x,
                     ax[2][kMaxAxisSegs - 1].x};
  const size_t nxy = (size_t)kp.n[0] * kp.n[1], nn = nxy * kp.n[2];
  for (int q = 0; q < ns[0] * ns[1] * ns[2]; ++q) {
    const int2 e[3] = {ax[0][q % ns[0]], ax[1][q / ns[0] % ns[1]], ax[2][q / (ns[0] * ns[1])]};
    const int id = brick_id(bd.ng, e[0].x, e[1].x, e[2].x);
    for (int j = bstart[id] + threadIdx.x; j < bstart[id + 1]; j += blockDim.x) {
      const uint32_t odd = __float_as_uint(fs[j].w);
      if (odd == 0u) continue;
      const uint32_t w = win[j];
      int lo[3], from[3], to[3];
      for (int a = 0; a < 3; ++a) {
        lo[a] = erpp_rec_lo(w, a) + e[a].y - (a == 2 ? z0 : 0);
        from[a] = max(lo[a], 0);
        to[a] = min(lo[a] + erpp_rec_nw(w, a), ext[a]);
      }
      for (int c = 0; c < 3; ++c) {
        const uint32_t k = (odd >> (3 * c)) & 7u;
        if (k == 0u) continue;
        const float v = k == 1u ? __int_as_float(0x7fffffff)
                                : __int_as_float(k == 2u ? 0x7f800000 : (int)0xff800000);
        for (int z = from[2]; z < to[2]; ++z)
          for (int y = from[1]; y < to[1]; ++y)
            for (int x = from[0]; x < to[0]; ++x)
              atomicAdd(S + c * nn + (b[2] + z) * nxy + (size_t)(b[1] + y) * kp.n[0] + b[0] + x,
                        v);
      }
    }
  }
}

// LP: lanes that stage a particle, each two neighbouring nodes per axis: 4 for
// windows of at most 7 nodes (at most 4 aligned pairs of nodes), else 8.
// axis: per axis a and group g the stretches of bricks that hold the home
// cells of the particles reaching the group's nodes (brick, first cell
// relative to the group); the last entry of the eight holds their number and
// 65536 / number, rounded up.
// ZS: planes of the region, 16, or 4 (planes z0 ..) of a dense one: there the
// block's four output tiles of 2 planes x 8 rows take four warps each, which
// share the tile's particles chunk by chunk and add their sums in order.
template <int LP, int ZS>
__device__ __forceinline__ void scatter_region(
    const erpp_kparams& kp, const erpp_brick_dims& bd, const int gg[3], int z0,
    const int2* __restrict__ axis, const float4* __restrict__ rec,
    const uint32_t* __restrict__ win, const float4* __restrict__ fs,
    const int32_t* __restrict__ bstart, const int32_t* __restrict__ bmax,
    const int32_t* __restrict__ skip, float* __restrict__ S, unsigned char* smem,
    ScatShared& sh) {
  constexpr int kTiles = ZS, kParts = kScatWarps / kTiles;  // 2 x 8-row tiles; warps of each
  unsigned char* const row0 = smem;  // [kListBatch + 1][kPitch]
  uint32_t* const mask = reinterpret_cast<uint32_t*>(row0 + (kListBatch + 1) * kPitch);
  unsigned char* const areas = reinterpret_cast<unsigned char*>(mask + kListBatch);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int skipped = skip ? __ldg(skip) : 0;  // looked at after the segments' loads
  const int b[3] = {gg[0] * kRegion, gg[1] * kRegion, gg[2] * kRegion + z0};
  const int ext[3] = {min(kRegion, kp.n[0] - b[0]), min(kRegion, kp.n[1] - b[1]),
                      min(ZS, kp.n[2] - b[2])};
  const uint32_t ext1 = 0x808080u | (uint32_t)(63 + ext[0]) | (uint32_t)(63 + ext[1]) << 8 |
                        (uint32_t)(63 + ext[2]) << 16;
  const int2* axx = axis + (size_t)gg[0] * kMaxAxisSegs;
  const int2* axy = axis + (size_t)(bd.ng[0] + gg[1]) * kMaxAxisSegs;
  const int2* axz = axis + (size_t)(bd.ng[0] + bd.ng[1] + gg[2]) * kMaxAxisSegs;
  const int2 nsx = axx[kMaxAxisSegs - 1], nsy = axy[kMaxAxisSegs - 1],
             nsz = axz[kMaxAxisSegs - 1];
  const int ns = min(nsx.x * nsy.x * nsz.x, kMaxSegs);
  const int K = (ns + kScatWarps - 1) / kScatWarps;  // segments per warp, at most 22

  if (tid == 0) {
    sh.maxbits = 0;
    sh.odd = 0;
  }
  if (tid < kPitch / 16)
    reinterpret_cast<uint4*>(row0 + kListBatch * kPitch)[tid] = make_uint4(0u, 0u, 0u, 0u);
  // Segment q: its brick's records, its first cell; returns the brick's
  // largest force component.
  auto describe = [&](int q, int& start, int& count, uint32_t& org) {
    const int r = (q * nsx.y) >> 16, rz = (r * nsy.y) >> 16;  // q / nsx, q / (nsx nsy)
    const int2 ex_ = axx[q - r * nsx.x], ey_ = axy[r - rz * nsy.x], ez_ = axz[rz];
    const int id = brick_id(bd.ng, ex_.x, ey_.x, ez_.x);
    start = bstart[id];
    count = bstart[id + 1] - start;
    org = (uint32_t)(ex_.y + 56) | (uint32_t)(ey_.y + 56) << 8 | (uint32_t)(ez_.y + 56 - z0) << 16;
    return bmax[id];
  };
  // Lane k describes the warp's k-th segment (the warps take turns, shifted
  // from turn to turn, so that each gets inner and outer bricks)
  int seg_s = 0, seg_c = 0, mx = 0;
  uint32_t seg_o = 0u;
  const int myq = lane * kScatWarps + ((warp + 5 * lane) & (kScatWarps - 1));
  if (lane < K && myq < ns) mx = describe(myq, seg_s, seg_c, seg_o);
  if (skipped) return;
  uint16_t* const mylist = reinterpret_cast<uint16_t*>(areas + warp * kArea);
  // queue[-1 - k]: the k-th member, its place in its segment (12 bits), the
  // warp's segment (5), its window's first node + 16 per axis (5 each)
  uint32_t* const queue = reinterpret_cast<uint32_t*>(areas + (warp + 1) * kArea);
  uint2* const dqueue = reinterpret_cast<uint2*>(mylist);  // dense regions: (record, window)

  // The members of the warp's segments, four segments at a time as one range,
  // 32 members a step; those that touch go into the warp's queue (while they
  // fit).
  int mine = 0;
  {
    for (int k = 0; k < K; k += 4) {
      int s0[4], e[4];
      uint32_t o[4];
      int tot = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // the member at position idx of the range is record idx + s0[i]
        s0[i] = __shfl_sync(0xffffffffu, seg_s, k + i) - tot;
        tot += __shfl_sync(0xffffffffu, seg_c, k + i);
        o[i] = __shfl_sync(0xffffffffu, seg_o, k + i);
        e[i] = tot;
      }
      for (int m0 = 0; m0 < tot; m0 += 32) {
        const int idx = m0 + lane;
        int j = s0[0], at0 = 0, sg = k;
        uint32_t og = o[0];
#pragma unroll
        for (int i = 1; i < 4; ++i) {
          const bool up = idx >= e[i - 1];
          j = up ? s0[i] : j;
          og = up ? o[i] : og;
          at0 = up ? e[i - 1] : at0;
          sg = up ? k + i : sg;
        }
        j += idx;
        const uint32_t w = idx < tot ? __ldg(&win[j]) : 0u;
        const bool t = idx < tot && touches(w, og, ext1);
        const uint32_t bal = __ballot_sync(0xffffffffu, t);
        const int at = mine + __popc(bal & ((1u << lane) - 1u));
        if (t && at < kArea / 4) {
          const uint32_t lo = window_lo(w, og) - 0x303030u;
          queue[-1 - at] = (uint32_t)(idx - at0) | (uint32_t)sg << 12 | (lo & 31u) << 17 |
                           (lo & 0x1f00u) << 14 | (lo >> 16) << 27;
        }
        mine += __popc(bal);
      }
    }
  }
  mx = __reduce_max_sync(0xffffffffu, (unsigned)mx);
  constexpr int kLong = 1 << 30;
  const bool seg_long = __any_sync(0xffffffffu, seg_c > kQueueMost);
  __syncthreads();  // maxbits is cleared
  if (lane == 0) {
    sh.cnt[warp] = mine | (seg_long ? kLong : 0);
    if (mx > 0) atomicMax(&sh.maxbits, mx);
  }
  __syncthreads();
  // The list: in one batch, or in several to which every warp gives an equal
  // part of its queue (a batch then holds total / nbatch + 16 at most).  Dense
  // regions, whose queues don't hold their members beside a batch's rows'
  // offsets, are listed again below.
  const int v = lane < kScatWarps ? sh.cnt[lane] & (kLong - 1) : 0;
  const int total = __reduce_add_sync(0xffffffffu, v);
  int nbatch = total <= kListBatch ? 1 : (total + kListBatch - 17) / (kListBatch - 16);
  const int room =
      nbatch == 1 ? kArea / 4 : (kArea - 2 * (total / nbatch + 16 + 16)) / 4;
  const bool dense =
      __any_sync(0xffffffffu, v > room || (lane < kScatWarps && sh.cnt[lane] >= kLong));
  DenseTab& tab = *reinterpret_cast<DenseTab*>(row0 + kDenseBatch * kPitch);
  int marks = 0, G = 32;
  // candidate idx of the range: its record, whether it touches, its window
  auto candidate = [&](int idx, int& j, uint32_t& lo) {
    if (idx >= tab.pre[ns]) return false;
    const int q = last_not_above(tab.pre, ns, idx);
    j = tab.start[q] + idx;
    const uint32_t w = __ldg(&win[j]), o = tab.org[q];
    lo = window_lo(w, o);
    return touches(w, o, ext1);
  };
  if (dense) {
    // more than one batch, or more than a warp can queue: the list is instead
    // in segment order, and every warp stages an equal share of each batch,
    // which it finds from the marks
    for (int q = tid; q < ns; q += kScatThreads) {
      int st, c;
      uint32_t o;
      describe(q, st, c, o);
      tab.start[q] = st;
      tab.org[q] = o;
      tab.pre[q] = c;
    }
    __syncthreads();
    if (warp == 0) warp_scan(tab.pre, ns, lane);
    __syncthreads();
    for (int q = tid; q < ns; q += kScatThreads) tab.start[q] -= tab.pre[q];
    const int C = tab.pre[ns];
    G = 32 * ((C + 32 * kMarks - 1) / (32 * kMarks));
    marks = (C + G - 1) / G;
    __syncthreads();
    for (int k = warp; k < marks; k += kScatWarps) {
      int m = 0;
      for (int i = 0; i < G; i += 32) {
        int j;
        uint32_t lo;
        m += __popc(__ballot_sync(0xffffffffu, candidate(k * G + i + lane, j, lo)));
      }
      if (lane == 0) tab.mark[k] = m;
    }
    __syncthreads();
    if (warp == 0) warp_scan(tab.mark, marks, lane);
    __syncthreads();
  }

  // factors scaled into the FP16 range: weights by 2^14 (at most 2^14), forces
  // by 2^(14 - ex) with the largest component below 2^ex
  const float fmx = __int_as_float(sh.maxbits);
  int ex = 0;
  frexpf(fmx, &ex);
  ex = max(ex, -100);
  const float sB = ldexpf(1.f, 14 - ex);

  const int tile = warp % kTiles, part = warp / kTiles;
  const int zp = tile % (ZS / 2), yh = tile / (ZS / 2);  // planes 2 zp, 2 zp + 1; rows 8 yh ..
  const int gr = lane >> 2, tq = lane & 3;
  Pair acc[3][2][2];
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int k = 0; k < 2; ++k) acc[c][h][k].v = 0ull;

  // batches of equal size, so that none leaves the warps a nearly empty chunk
  // (one, of none, where a brick around is long but nothing reaches these planes)
  if (dense) nbatch = max(1, (total + kDenseBatch - 1) / kDenseBatch);
  const int bsize = (total + nbatch - 1) / nbatch;

  // Stages members q0, q0 + 1, ... of the queue as rows p0, p0 + 1, ...: LP lanes a particle,
  // a pair of neighbouring nodes per axis each; the row cleared, then the
  // weights at the region's nodes.
  auto stage = [&](int q0, int p0, int nq) {
    const int ql = lane & (LP - 1);
    for (int i0 = 0; i0 < nq; i0 += 32 / LP) {
      const int i = i0 + lane / LP;
      const bool live = i < nq;
      const int qi = live ? i : i0;
      uint2 e;
      if (dense) {
        e = dqueue[qi];
      } else {
        const uint32_t m = queue[-1 - q0 - qi];
        e.x = (m & 4095u) + __shfl_sync(0xffffffffu, seg_s, (m >> 12) & 31u);
        e.y = (((m >> 17) & 31u) | (m >> 14 & 0x1f00u) | (m >> 27) << 16) + 0x303030u;
      }
      const float4 r = __ldg(&rec[e.x]);
      const float4 f = __ldg(&fs[e.x]);
      unsigned char* const row = row0 + (p0 + i) * kPitch;
      if (live) {
#pragma unroll
        for (int k = 0; k < (20 + LP - 1) / LP; ++k)
          if (LP == 4 || ql + k * LP < 20)
            *reinterpret_cast<uint4*>(row + 16 * (ql + k * LP)) = make_uint4(0u, 0u, 0u, 0u);
      }
      __syncwarp();
      const uint32_t w = __float_as_uint(r.w);
      const float t[3] = {r.x, r.y, r.z};
      float v[3][2];
      bool in[3];
      int at[3], lo[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        // the pair's first node in the region (even), and its window position
        lo[a] = (int)((e.y >> (8 * a)) & 255u) - 64;
        at[a] = (lo[a] & ~1) + 2 * ql;
        const int q = at[a] - lo[a];  // -1 at the least
        const int nw = erpp_rec_nw(w, a);
        const float k = (float)(erpp_rec_off(kp, w, a) + q);
        const Pair d = pair_of(k, k + 1.f) + pair_of(-t[a], -t[a]);
        const float2 e2 = parts(pair_of(-kp.beta[a], -kp.beta[a]) * d * d);
        v[a][0] = q >= 0 && q < nw ? erpp_ex2(e2.x) : 0.f;
        v[a][1] = q + 1 < nw ? erpp_ex2(e2.y) : 0.f;
        in[a] = live && q < nw && (unsigned)at[a] < 16u;
      }
      const Pair x01 = pair_of(v[0][0], v[0][1]) * pair_of(sB, sB);
      uint32_t h[3], l[3];
      split_pair(pair_of(f.x, f.x) * x01, h[0], l[0]);
      split_pair(pair_of(f.y, f.y) * x01, h[1], l[1]);
      split_pair(pair_of(f.z, f.z) * x01, h[2], l[2]);
      if (in[0]) {
        uint32_t* col = reinterpret_cast<uint32_t*>(row + 2 * at[0]);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          col[16 * c] = h[c];
          col[16 * c + 8] = l[c];
        }
      }
      float* const wt = reinterpret_cast<float*>(row + kRowW);
      if (in[1])
        *reinterpret_cast<float2*>(wt + at[1]) =
            make_float2(v[1][0] * 16384.f, v[1][1] * 16384.f);
      if (in[2]) *reinterpret_cast<float2*>(wt + 16 + at[2]) = make_float2(v[2][0], v[2][1]);
      if (live && ql == 0) {
        if (__float_as_uint(f.w) != 0u) sh.odd = 1;
        // the tiles whose rows and planes the window reaches: bit ZS / 2 yh + zp
        const int y1 = lo[1] + erpp_rec_nw(w, 1) - 1;
        const int za = max(lo[2], 0) >> 1, zb = min(lo[2] + erpp_rec_nw(w, 2) - 1, ZS - 1) >> 1;
        const uint32_t zm = (2u << zb) - (1u << za);
        mask[p0 + i] = (lo[1] < 8 ? zm : 0u) | (y1 >= 8 ? zm << (ZS / 2) : 0u);
      }
    }
  };

  for (int ib = 0; ib < nbatch; ++ib) {
    const int l0 = ib * bsize;
    int np = min(bsize, total - l0);
    // the warp's members of the batch
    if (!dense) {
      const int v = lane < kScatWarps ? sh.cnt[lane] : 0;
      const int from = nbatch == 1 ? 0 : v * ib / nbatch;
      const int share = (nbatch == 1 ? v : v * (ib + 1) / nbatch) - from;
      int incl = share;
#pragma unroll
      for (int o = 1; o < kScatWarps; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += u;
      }
      np = __shfl_sync(0xffffffffu, incl, kScatWarps - 1);
      stage(__shfl_sync(0xffffffffu, from, warp), __shfl_sync(0xffffffffu, incl - share, warp),
            __shfl_sync(0xffffffffu, share, warp));
    } else {
      // the warp's share: list positions [ra, rb)
      const int share = (np + kScatWarps - 1) / kScatWarps;
      const int ra = l0 + min(warp * share, np), rb = l0 + min((warp + 1) * share, np);
      if (ra < rb) {
        const int k = last_not_above(tab.mark, marks, ra);
        int at = tab.mark[k];
        for (int idx = k * G; at < rb && idx < tab.pre[ns]; idx += 32) {
          int j = 0;
          uint32_t lo = 0u;
          const bool t = candidate(idx + lane, j, lo);
          const uint32_t bal = __ballot_sync(0xffffffffu, t);
          const int p = at + __popc(bal & ((1u << lane) - 1u));
          if (t && p >= ra && p < rb) dqueue[p - ra] = make_uint2((uint32_t)j, lo);
          at += __popc(bal);
        }
      }
      __syncwarp();
      stage(0, ra - l0, rb - ra);
    }
    __syncthreads();
    // the warp's own particles, those that reach its rows and planes: their
    // rows' offsets in units of 16 bytes
    int cw = 0;
    for (int p0 = 0; p0 < np; p0 += 32) {
      const uint32_t m = p0 + lane < np ? mask[p0 + lane] : 0u;
      const bool t = (m >> tile) & 1u;
      const unsigned bal = __ballot_sync(0xffffffffu, t);
      if (t)
        mylist[cw + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)((p0 + lane) * (kPitch / 16));
      cw += __popc(bal);
    }
    if (lane < 16) mylist[cw + lane] = (uint16_t)(kListBatch * (kPitch / 16));  // the zero row
    __syncwarp();
    const unsigned char* const wty = row0 + kRowW + 4 * (8 * yh + gr);
    const unsigned char* const wtz = row0 + kRowW + 4 * (16 + 2 * zp);
    const unsigned btab = (unsigned)__cvta_generic_to_shared(row0) + ((lane >> 4) << 4);
    for (int c0 = 16 * part; c0 < cw; c0 += 16 * kParts) {
      const uint32_t pa = *reinterpret_cast<const uint32_t*>(mylist + c0 + 2 * tq);
      const uint32_t pb = *reinterpret_cast<const uint32_t*>(mylist + c0 + 8 + 2 * tq);
      const unsigned pk[4] = {(pa & 0xffffu) * 16u, (pa >> 16) * 16u, (pb & 0xffffu) * 16u,
                              (pb >> 16) * 16u};
      uint32_t ah[4], al[4];
#pragma unroll
      for (int k = 0; k < 4; k += 2) {
        const Pair y = pair_of(*reinterpret_cast<const float*>(wty + pk[k]),
                               *reinterpret_cast<const float*>(wty + pk[k + 1]));
        const float2 z0 = *reinterpret_cast<const float2*>(wtz + pk[k]);
        const float2 z1 = *reinterpret_cast<const float2*>(wtz + pk[k + 1]);
        split_pair(y * pair_of(z0.x, z1.x), ah[k], al[k]);
        split_pair(y * pair_of(z0.y, z1.y), ah[k + 1], al[k + 1]);
      }
      const unsigned addr = btab + 16u * mylist[c0 + (lane & 15)];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        uint32_t bh[4], bl[4];
        ldmatrix_x4_trans(bh, addr + (2 * c) * 32);
        ldmatrix_x4_trans(bl, addr + (2 * c + 1) * 32);
        // the chunk's own sums first (the tensor core truncates its sums; the
        // small products go first), then one rounded FP32 addition
        float d0[4], d1[4];
        mma_f16_zero(d0, al, bh[0], bh[1]);
        mma_f16_zero(d1, al, bh[2], bh[3]);
        mma_f16(d0, ah, bl[0], bl[1]);
        mma_f16(d1, ah, bl[2], bl[3]);
        mma_f16(d0, ah, bh[0], bh[1]);
        mma_f16(d1, ah, bh[2], bh[3]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          acc[c][0][k] = acc[c][0][k] + pair_of(d0[2 * k], d0[2 * k + 1]);
          acc[c][1][k] = acc[c][1][k] + pair_of(d1[2 * k], d1[2 * k + 1]);
        }
      }
    }
    if (ib + 1 < nbatch) __syncthreads();  // the rows are staged again
  }

  if (kParts > 1) {
    // the parts' sums, added in order by the first
    __syncthreads();
    Pair* const sums = reinterpret_cast<Pair*>(smem);  // [parts - 1][tiles][12][32]
    if (part > 0) {
      Pair* dst = sums + ((part - 1) * kTiles + tile) * 12 * 32 + lane;
#pragma unroll
      for (int k = 0; k < 12; ++k) dst[32 * k] = acc[k / 4][(k / 2) & 1][k & 1];
    }
    __syncthreads();
    for (int q = 0; q < kParts - 1 && part == 0; ++q) {
      const Pair* src = sums + (q * kTiles + tile) * 12 * 32 + lane;
#pragma unroll
      for (int k = 0; k < 12; ++k)
        acc[k / 4][(k / 2) & 1][k & 1] = acc[k / 4][(k / 2) & 1][k & 1] + src[32 * k];
    }
  }
  // a lane holds nodes (x, x + 1) of row gr of both planes
  const float inv = ldexpf(1.f, ex - 28);
  const size_t nxy = (size_t)kp.n[0] * kp.n[1], nn = nxy * kp.n[2];
  const int y = 8 * yh + gr;
  const bool pair = (kp.n[0] & 1) == 0 && (((uintptr_t)S) & 7) == 0;
  if (y < ext[1] && part == 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int x = 8 * h + 2 * tq;
#pragma unroll
      for (int z = 0; z < 2; ++z) {
        if (2 * zp + z >= ext[2] || x >= ext[0]) continue;
        float* d = S + (size_t)(b[2] + 2 * zp + z) * nxy + (size_t)(b[1] + y) * kp.n[0] + b[0] + x;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 v = parts(acc[c][h][z] * pair_of(inv, inv));
          if (pair) {
            *reinterpret_cast<float2*>(d + c * nn) = v;
          } else {
            d[c * nn] = v.x;
            if (x + 1 < ext[0]) d[c * nn + 1] = v.y;
          }
        }
      }
    }
  }
  if (sh.odd && total > (ZS == kRegion ? kOddRegion : kOddQuarter)) {
    __syncthreads();  // S has the block's finite sums
    add_odd_forces(kp, bd, gg[0], gg[1], gg[2], z0, ZS, axis, win, fs, bstart, S);
  }
}

// One block per region; the dense ones (the sort lists those near a dense brick)
// are k_brick_scatter_dense's.
template <int LP>
__global__ void __launch_bounds__(kScatThreads, 2) k_brick_scatter(
    erpp_kparams kp, erpp_brick_dims bd, const int32_t* __restrict__ dflag,
    const int2* __restrict__ axis, const float4* __restrict__ rec,
    const uint32_t* __restrict__ win, const float4* __restrict__ fs,
    const int32_t* __restrict__ bstart, const int32_t* __restrict__ bmax, float* __restrict__ S) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ ScatShared sh;
  const int gg[3] = {(int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z};
  scatter_region<LP, 16>(kp, bd, gg, 0, axis, rec, win, fs, bstart, bmax,
                         &dflag[(gg[2] * bd.ng[1] + gg[1]) * bd.ng[0] + gg[0]], S, smem, sh);
  // k_brick_scatter_dense, which this kernel runs beside, is done before this one is
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The dense regions by quarters of four planes, which the blocks take from a
// counter, ndense[1].  A kernel of its own, beside which k_brick_scatter starts
// at once: one kernel with both forms made the regions of a 512 x 256 x 256 box
// with 1M particles 1.6% slower (438 and 431 us), and taking the quarters by a fixed
// stride left clusters of 100k particles in 128^3 nodes at 400 - 470 us instead
// of 260 - 320.
template <int LP>
__global__ void __launch_bounds__(kScatThreads, 2) k_brick_scatter_dense(
    erpp_kparams kp, erpp_brick_dims bd, int32_t* __restrict__ ndense,
    const int32_t* __restrict__ dense, const int2* __restrict__ axis,
    const float4* __restrict__ rec, const uint32_t* __restrict__ win,
    const float4* __restrict__ fs, const int32_t* __restrict__ bstart,
    const int32_t* __restrict__ bmax, float* __restrict__ S) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ ScatShared sh;
  __shared__ int item;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int nd = 4 * *ndense;
  for (;;) {
    if (threadIdx.x == 0) item = atomicAdd(&ndense[1], 1);
    __syncthreads();
    const int it = item;
    if (it >= nd) break;
    const int g = dense[it >> 2], z0 = 4 * (it & 3);
    const int gg[3] = {g % bd.ng[0], (g / bd.ng[0]) % bd.ng[1], g / (bd.ng[0] * bd.ng[1])};
    if (gg[2] * kRegion + z0 < kp.n[2])
      scatter_region<LP, 4>(kp, bd, gg, z0, axis, rec, win, fs, bstart, bmax, nullptr, S, smem,
                            sh);
    __syncthreads();
  }
}

size_t scatter_smem() {
  return (size_t)(kListBatch + 1) * kPitch + (size_t)kListBatch * 4 +
         (size_t)kScatWarps * kArea;
}

// The stretches of bricks along an axis of n cells whose particles (windows
// starting at most hlo nodes below the home cell and ending at most hlo + 1
// above) can reach the nodes of group g: each stretch's brick and its first
// cell relative to the group's first node, periodic images included; the last
// entry holds their number.
void axis_segments(int n, int hlo, int g, int2* out) {
  const int b = g * kRegion, last = std::min(b + kRegion, n) - 1 + hlo;
  int k = 0;
  for (int j = b - hlo - 1; j <= last && k < kMaxAxisSegs - 1;) {
    const int m = j >= 0 ? j / n : -((-j + n - 1) / n);
    const int br = (j - m * n) >> 3;
    out[k].x = br;
    out[k].y = 8 * br + m * n - b;
    ++k;
    j = std::min(8 * br + 8, n) + m * n;
  }
  for (int i = k; i < kMaxAxisSegs - 1; ++i) out[i] = make_int2(-1, 0);
  out[kMaxAxisSegs - 1] = make_int2(k, 65536 / k + 1);
}

}  // namespace

namespace erpp {

// Whether the context's windows and options allow the brick kernels (windows
// of at most 10 nodes that start at most 4 below the cell: the record's
// fields; FP32, Gaussian source).
static bool bricks_possible(const erpp_ctx* c) {
  return !c->fp64 && c->kp.design == 4 && c->kp.weights != ERPP_W_PIC && !c->kp.kahan &&
         c->kp.xs <= 10 && c->kp.hlo <= 4;
}

// The brick kernels serve a call when the context's scatter mode is the
// default and the box has regions of 16^3 nodes for most SMs, or its particles
// are dense (a quarter of a particle per node, 16384 at least: the x/y-halo
// tiles then hold thousands of pieces each).  One source by bricks and by tiles:
// 64 regions, 16k particles (64^3) 51 and 44 us, but 64k 155 and 236 us; 125
// regions, 20k (80^3) 36 and 46; 180, 20k (96 x 96 x 80) 32 and 43; 512, 30k
// (128^3) 38 and 53 us.  One stretch inside is the tiles': uniform clouds with windows
// of 6 nodes at 0.06 to 0.11 particles per node, where tiles still sum up to 1024
// pieces in fixed point; a step by tiles and by bricks in 96^3 nodes, 53k particles
// 115 and 120 us, 88k 146 and 163 (128^3, 210k 247 and 276; 35k in 96^3 99 and 91, 133k
// 271 and 215).  The same number in clusters takes the tiles 914 us and the bricks 280
// (60k in 96^3), and the number alone doesn't tell which it is.
constexpr int64_t kRegionsLeast = 120;
static bool bricks_serve(const erpp_ctx* c, int64_t n) {
  if (!c->bk.cnt || c->scatter_mode != ERPP_SCATTER_MERGE || n <= 0) return false;
  const int64_t regions = c->bk.nbricks / 8;
  const double nodes = (double)c->kp.n[0] * c->kp.n[1] * c->kp.n[2];
  return regions >= kRegionsLeast || (n >= 16384 && (double)n >= 0.25 * nodes);
}

static size_t table_bytes(int nbricks) {
  return sizeof(int32_t) * (2 * (size_t)nbricks + 3 + (size_t)(nbricks / 8));
}

cudaError_t bricks_alloc_tables(erpp_ctx* c) {
  erpp_bricks& k = c->bk;
  if (!bricks_possible(c)) return cudaSuccess;
  int64_t ng = 1;
  for (int a = 0; a < 3; ++a) {
    k.dims.ng[a] = (c->kp.n[a] + kRegion - 1) / kRegion;
    ng *= k.dims.ng[a];
  }
  if (ng > (1 << 24) || k.dims.ng[1] > 65535 || k.dims.ng[2] > 65000) return cudaSuccess;
  k.nbricks = (int)(8 * ng);
  // cleared together: counts, force maxima, the numbers of further adjoint
  // chunks and of dense regions, the regions' dense flags
  cudaError_t e = cudaMalloc(&k.cnt, table_bytes(k.nbricks));
  if (e == cudaSuccess) e = cudaMalloc(&k.start, sizeof(int32_t) * ((size_t)k.nbricks + 4));
  if (e == cudaSuccess) e = cudaMalloc(&k.scan_tmp, sizeof(int32_t) * (k.nbricks / 4096 + 1));
  k.bmax = k.cnt ? k.cnt + k.nbricks : nullptr;
  k.nitems = k.cnt ? k.cnt + 2 * (size_t)k.nbricks : nullptr;
  k.ndense = k.cnt ? k.nitems + 1 : nullptr;
  k.dflag = k.cnt ? k.nitems + 3 : nullptr;
  if (e == cudaSuccess) e = cudaMalloc(&k.dense, sizeof(int32_t) * (size_t)(k.nbricks / 8));
  std::vector<int2> ax;
  for (int a = 0; a < 3; ++a)
    for (int g = 0; g < k.dims.ng[a]; ++g) {
      ax.resize(ax.size() + kMaxAxisSegs);
      axis_segments(c->kp.n[a], c->kp.hlo, g, ax.data() + ax.size() - kMaxAxisSegs);
    }
  if (e == cudaSuccess) e = cudaMalloc(&k.axis, sizeof(int2) * ax.size());
  if (e == cudaSuccess)
    e = cudaMemcpy(k.axis, ax.data(), sizeof(int2) * ax.size(), cudaMemcpyHostToDevice);
  return e;
}

void bricks_free_tables(erpp_ctx* c) {
  erpp_bricks& k = c->bk;
  cudaFree(k.cnt);
  cudaFree(k.start);
  cudaFree(k.scan_tmp);
  cudaFree(k.axis);
  cudaFree(k.dense);
  k.axis = nullptr;
  k.dense = k.ndense = k.dflag = nullptr;
  k.cnt = k.start = k.scan_tmp = k.bmax = k.nitems = nullptr;
}

bool stream_captures(cudaStream_t st) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &s) == cudaSuccess) return s != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return true;
}

}  // namespace erpp

// A former block: kept until the context's scratch goes, for the graphs that were
// captured with it.
struct erpp_brick_block {
  unsigned char* block;
  erpp_brick_block* next;
};

namespace erpp {

// The per-particle arrays for n particles, apart from the context's other scratch:
// made by the first call that sorts into bricks (76 bytes a particle, which a
// context that interpolates only, or in another halo mode, has no use for), so that
// an adjoint, which needs no scratch otherwise, leaves the other calls' alone.
// Where there is no memory for them the calls take the kernels that need none.
// Arrays that a capture has recorded stay in place when larger ones are made, of at
// least twice the size, so that all former ones together are no larger.
bool bricks_reserve(erpp_ctx* c, int64_t n) {
  erpp_bricks& k = c->bk;
  if (!bricks_serve(c, n)) return false;
  if (n <= k.cap) return true;
  if (k.refused > 0 && n >= k.refused) return false;
  erpp_brick_block* former = nullptr;
  size_t cap = (size_t)std::max<int64_t>(n, 1024);
  if (k.captured) {
    cap = std::max(cap, 2 * (size_t)k.cap);
    former = static_cast<erpp_brick_block*>(malloc(sizeof(erpp_brick_block)));
    if (!former) return false;
  } else {
    cudaFree(k.block);
    k.block = nullptr;
    k.cap = 0;
  }
  // one allocation: eleven of their own made a context's first call on 1M
  // particles 0.3 ms longer
  unsigned char* block = nullptr;
  size_t at = 0;
  auto place = [&](auto*& p, size_t count) {
    if (block) p = reinterpret_cast<std::remove_reference_t<decltype(p)>>(block + at);
    at += (count * sizeof(*p) + 255) & ~(size_t)255;
  };
  for (int pass = 0; pass < 2; ++pass) {
    at = 0;
    place(k.rec, cap);
    place(k.rec_in, cap);
    place(k.fs, cap);
    place(k.key, cap);
    place(k.items, cap / brick_chunk(c) + 1);
    place(k.pidx, cap);
    place(k.pbrick, cap);
    place(k.slot, cap);
    place(k.ord, cap);
    place(k.win, cap);
    if (pass == 1) break;
    if (cudaMalloc(&block, at) != cudaSuccess) {
      cudaGetLastError();
      free(former);
      k.refused = n;
      return false;
    }
  }
  if (former) {
    former->block = k.block;
    former->next = k.retired;
    k.retired = former;
    k.captured = false;
  }
  k.block = block;
  k.cap = (int64_t)cap;
  return true;
}

bool bricks_ready(erpp_ctx* c, int64_t n, cudaStream_t st) {
  if (!bricks_serve(c, n)) return false;
  const bool recorded = stream_captures(st);
  if (n > c->bk.cap && (recorded || !bricks_reserve(c, n))) return false;
  c->bk.captured |= recorded;
  return true;
}

void bricks_free(erpp_ctx* c) {
  erpp_bricks& k = c->bk;
  cudaFree(k.block);
  while (k.retired) {
    erpp_brick_block* r = k.retired;
    k.retired = r->next;
    cudaFree(r->block);
    free(r);
  }
  k.block = nullptr;
  k.cap = k.refused = 0;
  k.captured = false;
}

// Sorts n particles at x into bricks: bk.rec in order, bk.slot each particle's
// place (-1: invalid position), bk.start the bricks' ranges; for the adjoint bk.ord
// and its further chunks.  What only the adjoint reads keeps the order of arrival
// within a brick, and is sorted by a launch less.
cudaError_t brick_sort(erpp_ctx* c, int64_t n, const double* const x[3], bool for_source,
                       bool for_adjoint, cudaStream_t st) {
  erpp_bricks& k = c->bk;
  const int nb = k.nbricks;
  cudaError_t e = cudaMemsetAsync(k.cnt, 0, table_bytes(nb), st);
  if (e != cudaSuccess) return e;
  const unsigned blocks = (unsigned)((n + 255) / 256);
  // the records in order of arrival: where the forces go later
  float4* rec_tmp = for_source ? k.fs : k.rec;
  const AdjOrder adj = {for_adjoint ? k.ord : nullptr, k.nitems, k.items, brick_tile(c),
                        brick_chunk(c)};
  ++c->launches;
  e = erpp_launch_pdl(k_brick_count, dim3(blocks), dim3(256), 0, st, 0u, c->kp, k.dims, n, x[0],
                      x[1], x[2], k.rec_in, k.key, k.cnt, c->err);
  if (e != cudaSuccess) return e;
  if (nb <= kBrickScanOne) {
    ++c->launches;
    e = erpp_launch_pdl(k_brick_scan, dim3((unsigned)((nb + 4095) / 4096)), dim3(1024), 0, st, 0u, (const int32_t*)k.cnt,
                        k.start, nb);
  } else {
    e = launch_scan(c, k.cnt, k.start, k.scan_tmp, nb, st);
  }
  if (e != cudaSuccess) return e;
  ++c->launches;
  e = erpp_launch_pdl(k_brick_place, dim3(blocks), dim3(256), 0, st, 0u, n, (const int2*)k.key,
                      (const float4*)k.rec_in, (const int32_t*)k.start, rec_tmp, k.pidx, k.pbrick,
                      k.slot, for_source ? AdjOrder{} : adj);
  if (e != cudaSuccess || !for_source) return e;
  ++c->launches;
  return erpp_launch_pdl(k_brick_order, dim3(blocks), dim3(256), 0, st, 0u, n, nb,
                         (const int32_t*)k.pidx, (const int32_t*)k.pbrick, (const float4*)rec_tmp,
                         (const int32_t*)k.start, k.rec,
                         k.win, k.slot, adj, c->kp, k.dims, k.ndense, k.dense, k.dflag);
}

cudaError_t brick_forces(erpp_ctx* c, int64_t n, const double* const D[3], float scale,
                         cudaStream_t st) {
  erpp_bricks& k = c->bk;
  ++c->launches;
  k_brick_forces<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(
      c->kp, n, D[0], D[1], D[2], scale, k.rec, k.key, k.slot, k.fs, k.bmax);
  return cudaGetLastError();
}

cudaError_t brick_scatter(erpp_ctx* c, float* S, cudaStream_t st) {
  erpp_bricks& k = c->bk;
  const size_t sm = scatter_smem();
  const bool four = c->kp.xs <= 7;
  auto kern = four ? k_brick_scatter<4> : k_brick_scatter<8>;
  auto dkern = four ? k_brick_scatter_dense<4> : k_brick_scatter_dense<8>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(dkern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  c->launches += 2;
  c->route |= ERPP_ROUTE_SOURCE;
  constexpr int kResident = 2 * ERPP_SMS;
  dkern<<<kResident, kScatThreads, sm, st>>>(c->kp, k.dims, k.ndense, k.dense, k.axis, k.rec, k.win,
                                       k.fs, k.start, k.bmax, S);
  // started beside the dense regions' kernel: its blocks wait for that one last
  const dim3 grid((unsigned)k.dims.ng[0], (unsigned)k.dims.ng[1], (unsigned)k.dims.ng[2]);
  return erpp_launch_pdl(kern, grid, dim3(kScatThreads), sm, st, 0, c->kp, k.dims, k.dflag, k.axis,
                         k.rec, k.win, k.fs, k.start, k.bmax, S);
}

}  // namespace erpp
