// erpp_bricks_adjoint.cu -- the adjoint contractions of erpp_adjoint.cu for
// FP32 grids from brick-sorted particles, with the same FP32 arithmetic (every
// product and sum in the same order, so the results are the same bit for bit).
//
// A block serves the particles of one tile of cells (one range of the sorted
// records): it stages the tile's field with a halo as wide as a window on all
// sides (one TMA box; 16-byte copies where the box wraps around the periodic
// box; word by word where rows are not 16-byte aligned).  A warp takes two
// particles at a time: their weights and derivative weights into shared memory,
// 16 lanes to a particle, then each lane a (y, z) row of the window, walked along
// x in 16-byte loads.  The warps meet for the field only: with the weights of 40
// particles written by the whole block between two barriers the warps waited for
// one another, and 100k particles with windows of 9 nodes in 128^3 nodes took
// 207 us instead of 170.  Shared memory then bounds it, and two blocks per SM.
//
// The warp-per-particle kernel reads the field from global memory, each lane
// its own row, so that every load touches 32 lines, wraps every node index by a
// 64-bit remainder, and evaluates windows, distances and the weights' constants
// in FP64, whose pipe is narrow: 820 us for 100k particles with windows of 9
// nodes.  Here a window row is three conflict-free 16-byte shared loads (rows
// of 28 words), and the only FP64 operation is the position's product with
// N / L: the distances come from its bits by integer arithmetic.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_runtime.h>

#include <string.h>

#include <algorithm>

#include "erpp_async.cuh"
#include "erpp_internal.cuh"

namespace {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;

// Tile and staged box of a window class.  HL: nodes staged below the tile in y
// and z (x: 4, so that the box starts on 16 bytes); NW: longest window.  A tile
// is TB consecutive bricks of a group; kChunk particles of it per block (100k
// particles in 128^3 nodes, 49 a tile: 189 us with chunks of 48, 170 with 64 or
// 96, which dense tiles then share among more blocks than with longer ones).
struct Geo7 {  // windows of at most 7 nodes that start at most 3 below the cell
  static constexpr int TB = 4, PX = 24, NY = 23, NZ = 15, HL = 3, NW = 7;
  static constexpr int kChunk = 96;
};
struct Geo10 {  // at most 10 nodes, 4 below the cell
  static constexpr int TB = 2, PX = 28, NY = 17, NZ = 17, HL = 4, NW = 10;
  static constexpr int kChunk = 96;
};

// A particle's row in shared memory: x-weights by staged column from a multiple
// of 4, y- and z-weights, each with the derivative weights beside; then the
// window's place and size, and the co-vector.
template <class G>
struct Row {
  static constexpr int kX = 0, kDX = 16, kY = 32, kDY = kY + G::NW, kZ = kDY + G::NW,
                       kDZ = kZ + G::NW, kMeta = (kDZ + G::NW + 3) & ~3, kRow = kMeta + 8;
};

struct AdjArgs {
  const int32_t* ord;  // particle of each record
  const double* x[3];
  const double* v[3];  // co-vector
  double* val[3];      // alpha G (optional)
  double* der[3];      // alpha h (+ shear v_x on y)
  double alpha, shear;
  float raw1, sig2, dx[3];  // weights' constants in FP32
};

// Sums v[k] over the warp's lanes; the lanes with lane >> 2 == k get the sum of
// v[k].  Each of the first three steps halves the values a lane carries.
__device__ __forceinline__ float warp_sum8(const float (&v)[8], int lane) {
  float a[4], b[2];
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float keep = h16 ? v[4 + k] : v[k], send = h16 ? v[k] : v[4 + k];
    a[k] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const float keep = h8 ? a[2 + k] : a[k], send = h8 ? a[k] : a[2 + k];
    b[k] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
  }
  float s = (h4 ? b[1] : b[0]) + __shfl_xor_sync(0xffffffffu, h4 ? b[0] : b[1], 4);
  s += __shfl_xor_sync(0xffffffffu, s, 2);
  s += __shfl_xor_sync(0xffffffffu, s, 1);
  return s;
}

__device__ __forceinline__ int wrap_mod(int j, int n) {
  const int r = j % n;
  return r < 0 ? r + n : r;
}
// The same without a division where j is at most one period off.
__device__ __forceinline__ int wrap_near(int j, int n) {
  const int r = j < 0 ? j + n : (j >= n ? j - n : j);
  return (unsigned)r < (unsigned)n ? r : wrap_mod(j, n);
}

// Copies of the tile's box by the whole block where one TMA box cannot: 16 bytes
// a thread (nx a multiple of 4, u 16-byte aligned; no four words straddle the
// box's end), else word by word.  Both are calls: inlined, they made the kernel of
// 100k particles with windows of 9 nodes 20 us longer.
template <class G>
__device__ __noinline__ void stage_rows(const erpp_kparams& kp, const float* __restrict__ u,
                                         float* field, const int b[3]) {
  const size_t nn = (size_t)kp.n[0] * kp.n[1] * kp.n[2];
  const int gx0 = wrap_mod(b[0] - 4, kp.n[0]);
  constexpr int kQ = G::PX / 4;
  for (int i = threadIdx.x; i < 3 * G::NZ * G::NY * kQ; i += kThreads) {
    const int r = i / kQ, q = i - r * kQ;
    const int cz = r / G::NY, y = r - cz * G::NY;
    const int c = cz / G::NZ, z = cz - c * G::NZ;
    const int gy = wrap_near(b[1] - G::HL + y, kp.n[1]), gz = wrap_near(b[2] - G::HL + z, kp.n[2]);
    const int gx = wrap_near(gx0 + 4 * q, kp.n[0]);
    cp_async16(field + 4 * i, u + c * nn + ((size_t)gz * kp.n[1] + gy) * kp.n[0] + gx);
  }
}
// A lane keeps its column.  Its instructions bound this form (a row is 24 or 28
// words and as many index sums): with a remainder per index instead of
// wrap_near a box of 250 x 251 x 253 nodes with 16k particles took 847 us, now 604.
template <class G>
__device__ __noinline__ void stage_words(const erpp_kparams& kp, const float* __restrict__ u, float* field,
                            const int b[3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane >= G::PX) return;
  const float* const col = u + wrap_mod(b[0] - 4 + lane, kp.n[0]);
#pragma unroll 4
  for (int r = warp; r < 3 * G::NZ * G::NY; r += kWarps) {
    const int cz = r / G::NY, y = r - cz * G::NY;
    const int c = cz / G::NZ, z = cz - c * G::NZ;
    const int gy = wrap_near(b[1] - G::HL + y, kp.n[1]), gz = wrap_near(b[2] - G::HL + z, kp.n[2]);
    cp_async4(field + r * G::PX + lane,
              col + (((size_t)c * kp.n[2] + gz) * kp.n[1] + gy) * kp.n[0]);
  }
}

// RN(k - f) in FP32, f the fractional part of s >= 0 and k an integer of at most
// 16: from the bits of s, without FP64 arithmetic (which serves where s is below
// 1/32).
__device__ __forceinline__ float distance(double s, int k) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(s);
  const int sh = 1075 - (int)((b >> 52) & 0x7ffu);
  if (sh > 57 || sh < 0) return (float)((double)k - (s - floor(s)));
  const unsigned long long m = (b & 0xfffffffffffffull) | (1ull << 52);
  const long long v = ((long long)k << sh) - (long long)(m & ((1ull << sh) - 1ull));
  return __ll2float_rn(v) * __int_as_float((127 - sh) << 23);
}

// Sum over 16 lanes by halves (8, 4, 2, 1), the order of a warp's butterfly
// whose upper half holds zeros.
__device__ __forceinline__ float half_sum(float v) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <class G>
__global__ void __launch_bounds__(kThreads, 2) k_brick_adjoint(
    erpp_kparams kp, erpp_brick_dims bd, const float* __restrict__ u,
    const __grid_constant__ CUtensorMap tmap, int use_tma, int rows_ok, int nextra,
    const float4* __restrict__ rec, const int32_t* __restrict__ bstart,
    const int32_t* __restrict__ nitems, const int2* __restrict__ items, AdjArgs ag, int64_t n,
    const int32_t* __restrict__ slot, int nbricks, uint32_t* err) {
  using T = Row<G>;
  constexpr int PL = G::PX * G::NY, CS = PL * G::NZ;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ __align__(8) uint64_t stall_bar;  // debug_stall only: never completed
  float* const field = reinterpret_cast<float*>(smem);
  constexpr int kField = 3 * CS;
  float* const tables = field + kField + 16;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned phase = 0;
  if (tid == 0) {
    mbar_init(&bar, 1);
    if (kp.debug_stall) mbar_init(&stall_bar, 1);
  }
  __syncthreads();
  // Particles without a record (invalid positions): zeros, as their windows are
  // empty.  One block looks for them, when the records are fewer than the
  // particles.
  if (blockIdx.x == gridDim.x - 1 && bstart[nbricks] < n) {
    for (int64_t i = tid; i < n; i += kThreads) {
      if (slot[i] >= 0) continue;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        if (ag.val[a]) ag.val[a][i] = 0.0;
        ag.der[a][i] = 0.0;
      }
    }
  }
  // the first blocks: the further chunks of dense tiles, in turn; the others: a
  // tile's first chunk each
  const bool extra = (int)blockIdx.x < nextra;
  const int nit = extra ? *nitems : 1;
  for (int it = extra ? (int)blockIdx.x : 0; it < nit; it += nextra) {
    const int tile = extra ? items[it].x : (int)blockIdx.x - nextra;
    const int j0 = extra ? items[it].y : bstart[tile * G::TB];
    const int cnt = min(bstart[tile * G::TB + G::TB] - j0, G::kChunk);
    if (cnt <= 0) break;
    int b[3];
    {
      constexpr int TG = 8 / G::TB;  // tiles of a group
      int g = tile / TG;
      const int h = tile - g * TG;
      b[0] = (g % bd.ng[0]) * 16;
      g /= bd.ng[0];
      b[1] = (g % bd.ng[1]) * 16 + (G::TB == 2 ? 8 * (h & 1) : 0);
      b[2] = (g / bd.ng[1]) * 16 + (G::TB == 2 ? 8 * (h >> 1) : 8 * h);
    }
    // the field
    const int x0 = b[0] - 4, y0 = b[1] - G::HL, z0 = b[2] - G::HL;
    const bool tma = use_tma && x0 >= 0 && x0 + G::PX <= kp.n[0] && y0 >= 0 &&
                     y0 + G::NY <= kp.n[1] && z0 >= 0 && z0 + G::NZ <= kp.n[2];
    if (tma) {
      if (tid == 0) {
        // a block's next further chunk: its box lands where the tile before was
        // staged, by the generic proxy perhaps, and read; the block's barrier and
        // this fence put those accesses before the copy's
        if (extra && it != (int)blockIdx.x) fence_proxy_async_shared();
        mbar_expect_tx(&bar, (unsigned)(kField * 4));
        tma_load_4d(field, &tmap, &bar, x0, y0, z0, 0);
      }
    } else if (rows_ok) {
      stage_rows<G>(kp, u, field, b);
    } else {
      stage_words<G>(kp, u, field, b);
    }
    // A warp takes two particles at a time: their weights, then their sums.  The
    // block meets only for the field.
    bool waited = false;
    float* const table = tables + warp * 2 * T::kRow;
    for (int p0 = 2 * warp;; p0 += 2 * kWarps) {
      const int np = min(2, cnt - p0);
      // the weights: 16 lanes to a particle, a node of the window each
      const int ql = lane & 15;
      if (np > 0) {
        const int p = min(lane >> 4, np - 1);
        const int j = j0 + p0 + p;
        const uint32_t w = __float_as_uint(__ldg(&rec[j].w));
        const int pi = ag.ord[j];
        double xp[3];
        float vp[3];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          xp[a] = ag.x[a][pi];
          vp[a] = (float)ag.v[a][pi];
        }
        // the brick in the tile (its place among the bricks' ranges)
        int brick = 0;
#pragma unroll
        for (int k = 1; k < G::TB; ++k) brick += j >= bstart[tile * G::TB + k] ? 1 : 0;
        float* const row = table + p * T::kRow;
        const int sx = erpp_rec_lo(w, 0) + 4 + 8 * (brick & 1);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const int nw = erpp_rec_nw(w, a), off = erpp_rec_off(kp, w, a);
          const double s = __dmul_rn(xp[a], kp.inv_dx[a]);
          const float sig2 = ag.sig2, dxa = ag.dx[a];
          float wv = 0.f, d = 0.f;
          if (ql < nw) {
            d = distance(s, off + ql) * dxa;  // signed distance x_j - x_p
            wv = ag.raw1 * expf(-(d * d) / (2.f * sig2));
          }
          // lanes beyond the window divide ones: a zero takes a division's slow way
          const bool idle = ql >= nw;
          float dwv;
          if (kp.normalize) {
            const float sum = half_sum(wv);
            wv = (idle ? 1.f : wv) / (dxa * sum);
            const float mean = dxa * half_sum(wv * d);  // dx sum_k w_k d_k
            dwv = (idle ? 1.f : wv * (d - mean)) / sig2;
          } else {
            dwv = (idle ? 1.f : wv * d) / sig2;
          }
          if (!idle) {
            row[(a == 0 ? T::kX + (sx & 3) : (a == 1 ? T::kY : T::kZ)) + ql] = wv;
            row[(a == 0 ? T::kDX + (sx & 3) : (a == 1 ? T::kDY : T::kDZ)) + ql] = dwv;
          }
        }
        if (ql == 0) {
          // the window's first staged word, its columns from a multiple of 4, and
          // r / ny for r < 128 as r (65536 / ny + 1) / 65536
          const int sy = erpp_rec_lo(w, 1) + G::HL + (G::TB == 4 ? 8 * (brick >> 1) : 0);
          const int nwx = erpp_rec_nw(w, 0), ny = erpp_rec_nw(w, 1);
          *reinterpret_cast<int4*>(row + T::kMeta) =
              make_int4(((erpp_rec_lo(w, 2) + G::HL) * G::NY + sy) * G::PX + (sx & ~3),
                        (int)(((1u << nwx) - 1u) << (sx & 3)), ny | (65536 / ny + 1) << 4,
                        erpp_rec_nw(w, 2));
#pragma unroll
          for (int a = 0; a < 3; ++a) row[T::kMeta + 4 + a] = vp[a];
        }
      }
      if (!waited) {
        // one thread waits (bounded) for the field; the block goes on or gives up
        // as a whole
        if (!tma) cp_async_wait_all();
        int timed_out = 0;
        if (tma && tid == 0) {
          bool ok = mbar_wait_ns(&bar, phase, kp.wait_ns);
          if (!ok) {
            mbar_wait_ns(&bar, phase, kp.wait_ns);  // once more for the copy in flight
          } else if (kp.debug_stall) {
            ok = mbar_wait_ns(&stall_bar, 0, kp.wait_ns);  // nothing arrives: runs out
          }
          if (!ok) {
            erpp_set_err(err, ERPP_ERRBIT_TIMEOUT);
            timed_out = 1;
          }
        }
        if (__syncthreads_or(timed_out)) return;
        // the phase has completed: every thread observes it, which returns at once
        if (tma) {
          if (tid != 0) mbar_try_wait(&bar, phase);
          phase ^= 1u;
        }
        waited = true;
      }
      if (np <= 0) break;
      __syncwarp();
      for (int p = 0; p < np; ++p) {
        float* const row = table + p * T::kRow;
        const int4 meta = *reinterpret_cast<const int4*>(row + T::kMeta);
        const float v0 = row[T::kMeta + 4], v1 = row[T::kMeta + 5], v2 = row[T::kMeta + 6];
        const unsigned cols = (unsigned)meta.y;  // the window's columns, from the first load
        const int ny = meta.z & 15, per = meta.z >> 4, rows = ny * meta.w;
        float g0 = 0.f, g1 = 0.f, g2 = 0.f, h0 = 0.f, h1 = 0.f, h2 = 0.f;
        for (int r = lane; r < rows; r += 32) {
          const int kz = (r * per) >> 16, ky = r - kz * ny;
          const float* f = field + meta.x + kz * PL + ky * G::PX;
          float a0 = 0.f, a1 = 0.f, a2 = 0.f, b0 = 0.f, b1 = 0.f, b2 = 0.f;
#pragma unroll
          for (int k = 0; k < (G::NW + 6) / 4; ++k) {
            if ((cols >> (4 * k)) == 0u) break;
            const float4 q0 = *reinterpret_cast<const float4*>(f + 4 * k);
            const float4 q1 = *reinterpret_cast<const float4*>(f + CS + 4 * k);
            const float4 q2 = *reinterpret_cast<const float4*>(f + 2 * CS + 4 * k);
            const float4 wx = *reinterpret_cast<const float4*>(row + T::kX + 4 * k);
            const float4 dx = *reinterpret_cast<const float4*>(row + T::kDX + 4 * k);
            auto node = [&](int m, float u0, float u1, float u2, float w, float dw) {
              if ((cols >> (4 * k + m)) & 1u) {  // the same in every lane
                a0 = fmaf(u0, w, a0);
                a1 = fmaf(u1, w, a1);
                a2 = fmaf(u2, w, a2);
                b0 = fmaf(u0, dw, b0);
                b1 = fmaf(u1, dw, b1);
                b2 = fmaf(u2, dw, b2);
              }
            };
            node(0, q0.x, q1.x, q2.x, wx.x, dx.x);
            node(1, q0.y, q1.y, q2.y, wx.y, dx.y);
            node(2, q0.z, q1.z, q2.z, wx.z, dx.z);
            node(3, q0.w, q1.w, q2.w, wx.w, dx.w);
          }
          const float wy = row[T::kY + ky], wz = row[T::kZ + kz];
          const float wyz = wy * wz, dyz = row[T::kDY + ky] * wz, ydz = wy * row[T::kDZ + kz];
          const float av = fmaf(a2, v2, fmaf(a1, v1, a0 * v0));
          const float bv = fmaf(b2, v2, fmaf(b1, v1, b0 * v0));
          g0 = fmaf(a0, wyz, g0);
          g1 = fmaf(a1, wyz, g1);
          g2 = fmaf(a2, wyz, g2);
          h0 = fmaf(bv, wyz, h0);
          h1 = fmaf(av, dyz, h1);
          h2 = fmaf(av, ydz, h2);
        }
        const float v[8] = {g0, g1, g2, h0, h1, h2, 0.f, 0.f};
        const float sum = warp_sum8(v, lane);
        // the sums replace the weights, which every lane is done with
        __syncwarp();
        if ((lane & 3) == 0) row[lane >> 2] = sum;
      }
      __syncwarp();
      if (lane < 6 * np) {
        const int p = lane >= 6 ? 1 : 0, q = lane - 6 * p;
        const float sum = table[p * T::kRow + q];
        const int i = ag.ord[j0 + p0 + p];
        if (q < 3) {
          double* const to = q == 0 ? ag.val[0] : (q == 1 ? ag.val[1] : ag.val[2]);
          if (to) to[i] = ag.alpha * (double)sum;
        } else if (q == 4) {
          ag.der[1][i] = ag.alpha * (double)sum + ag.shear * ag.v[0][i];
        } else {
          (q == 3 ? ag.der[0] : ag.der[2])[i] = ag.alpha * (double)sum;
        }
      }
      __syncwarp();  // the table is written again
    }
    // a block that took a tile's first chunk is done (without further chunks' blocks,
    // nextra = 0, the loop has no step)
    if (!extra) break;
    __syncthreads();  // the field is written again
  }
}

template <class G>
cudaError_t launch(erpp_ctx* c, const float* u, int64_t n, const AdjArgs& ag, cudaStream_t st) {
  const erpp_kparams& kp = c->kp;
  erpp_bricks& k = c->bk;
  auto kern = k_brick_adjoint<G>;
  const size_t sm = sizeof(float) * (3 * (size_t)G::NZ * G::NY * G::PX + 16 +
                                     2 * kWarps * (size_t)Row<G>::kRow);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (e != cudaSuccess) return e;
  CUtensorMap map;
  memset(&map, 0, sizeof(map));
  const int rows_ok = (kp.n[0] & 3) == 0 && (((uintptr_t)u) & 15) == 0;
  const int box[3] = {G::PX, G::NY, G::NZ};
  const int use_tma = rows_ok && erpp::field_box_map(kp, u, box, &map) ? 1 : 0;
  const int nextra = (int)std::min<int64_t>(n / G::kChunk, 4 * ERPP_SMS);
  ++c->launches;
  kern<<<(unsigned)(k.nbricks / G::TB + nextra), kThreads, sm, st>>>(
      kp, k.dims, u, map, use_tma, rows_ok, nextra, k.rec, k.start, k.nitems, k.items, ag, n,
      k.slot, k.nbricks, c->err);
  return cudaGetLastError();
}

bool short_windows(const erpp_ctx* c) { return c->kp.xs <= 7 && c->kp.hlo <= 3; }

}  // namespace

namespace erpp {

int brick_tile(const erpp_ctx* c) { return short_windows(c) ? Geo7::TB : Geo10::TB; }
int brick_chunk(const erpp_ctx* c) { return short_windows(c) ? Geo7::kChunk : Geo10::kChunk; }

// Whether n particles pay for the sort and for staging every tile with its halo.
// The warp-per-particle kernel takes 4.6 - 9 ns a particle, whatever the box; here
// the sort's three launches cost ten us, and a tile that holds any particle as much
// as about six (its box by TMA or in 16-byte copies) or twenty (word by word, rows
// that are no multiple of 16 bytes).  Uniform clouds, windows of 6 nodes and of 9,
// by warps and by bricks in us: 96 x 96 x 80 nodes, 4k particles 32 and 37, 56 and
// 42, 5k 40 and 37, 68 and 44; 128^3, 6k 46 and 48, 80 and 70, 8k 52 and 49, 91 and
// 73; 256^3, 34k (0.002 a node) 178 and 204, 327 and 337, 50k (0.003) 252 and 220.
// Odd rows: 90 x 83 x 85, 12k 64 and 68, 30k 146 and 108; 181 x 122 x 95, 31k (0.015
// a node) 152 and 150, 201 and 200; 250 x 251 x 253, 0.015 a node 1089 and 896, 1619
// and 1282.
bool bricks_pay_adjoint(const erpp_ctx* c, int64_t n, const void* F) {
  const bool rows_ok = (c->kp.n[0] & 3) == 0 && ((uintptr_t)F & 15) == 0;
  const double nodes = (double)c->kp.n[0] * c->kp.n[1] * c->kp.n[2];
  return rows_ok ? n >= 5000 && (double)n >= 0.0035 * nodes
                 : n >= 14000 && (double)n >= 0.015 * nodes;
}

cudaError_t brick_adjoint(erpp_ctx* c, int64_t n, const double* const x[3], const float* F,
                          const double* const v[3], double alpha, double shear_coef,
                          double* const outv[3], double* const outx[3], cudaStream_t st) {
  AdjArgs ag = {};
  ag.ord = c->bk.ord;
  ag.alpha = alpha;
  ag.shear = shear_coef;
  ag.raw1 = (float)c->kp.raw_norm1;
  ag.sig2 = (float)c->kp.sig2;
  for (int a = 0; a < 3; ++a) {
    ag.x[a] = x[a];
    ag.v[a] = v[a];
    ag.val[a] = outv ? outv[a] : nullptr;
    ag.der[a] = outx[a];
    ag.dx[a] = (float)c->kp.dx[a];
  }
  return short_windows(c) ? launch<Geo7>(c, F, n, ag, st) : launch<Geo10>(c, F, n, ag, st);
}

}  // namespace erpp
