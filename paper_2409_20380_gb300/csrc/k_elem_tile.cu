// Tiled element-by-element product for meshes without hex patches: linear tets in any order and quadratic tets.
// The plain kernels add every element's corner sums into global memory by FP32 atomics, and those atomics bound
// them (0.6e12 scalar adds a second: 8 cases on 386,370 linear tets 63 us, 16 cases on 786,432 quadratic ones 621
// us).  Here a block takes a run of consecutive elements, sums its nodes in shared memory and adds each node once.
//
// The tiles' node lists and the elements' tile-local corner ids are built on the GPU at mesh creation.  Tile sums
// are 32-bit fixed point added by native integer atomics (an FP32 atomic add on shared memory is a
// compare-and-swap loop): per tile and case scaled by 2^(30 - E), 2^E above (|aM| abs_m + |aK| abs_k) max |p| over
// the tile's nodes, which bounds every partial sum of a row; a contribution is rounded to 2^-31 of that bound.  A
// tile whose bound is not finite adds its elements' sums to global memory in FP32 instead, so infinities and NaN
// reach the rows they belong to.
#include <type_traits>

#include "elem_ops.cuh"

namespace fem {

namespace {

constexpr int kSortMax = 1024;      // corner references of a tile (sorted in shared memory)

// One block a tile: its distinct nodes, sorted (the entries carry the node's free-DOF bits at 28-30), and each
// reference's index among them.  stats: [0] largest count, [1] sum of the counts.
template <int NPE>
__global__ void __launch_bounds__(kBlock) k_tile_nodes(int64_t E, int per_tile, const int32_t* __restrict__ conn,
                                                       const uint8_t* __restrict__ fm, int* __restrict__ count,
                                                       int* __restrict__ nodes, uint16_t* __restrict__ loc,
                                                       unsigned long long* __restrict__ stats) {
  __shared__ int key[kSortMax];
  __shared__ int uniq[kSortMax];
  __shared__ int wsum[kBlock / 32];
  const int64_t e0 = (int64_t)blockIdx.x * per_tile;
  const int refs = (int)min((int64_t)per_tile, E - e0) * NPE;
  const int32_t* src = conn + e0 * NPE;
  for (int i = threadIdx.x; i < kSortMax; i += kBlock) key[i] = i < refs ? src[i] : INT32_MAX;
  __syncthreads();
  for (int k = 2; k <= kSortMax; k <<= 1)          // bitonic sort
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < kSortMax; i += kBlock) {
        const int o = i ^ j;
        if (o > i) {
          const int a = key[i], b = key[o];
          if ((a > b) == ((i & k) == 0)) key[i] = b, key[o] = a;
        }
      }
      __syncthreads();
    }
  // each thread owns four consecutive keys; first occurrences are ranked by a block scan
  constexpr int PER = kSortMax / kBlock;
  int first[PER], mine = 0;
#pragma unroll
  for (int u = 0; u < PER; ++u) {
    const int i = threadIdx.x * PER + u;
    first[u] = i < refs && (i == 0 || key[i] != key[i - 1]);
    mine += first[u];
  }
  int pre = mine;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, pre, o);
    if (lane >= o) pre += v;
  }
  if (lane == 31) wsum[warp] = pre;
  __syncthreads();
  int rank = pre - mine, total = 0;
  for (int w = 0; w < kBlock / 32; ++w) {
    if (w < warp) rank += wsum[w];
    total += wsum[w];
  }
  if (threadIdx.x == 0) {
    count[blockIdx.x] = total;
    atomicMax(stats, (unsigned long long)total);
    atomicAdd(stats + 1, (unsigned long long)total);
  }
#pragma unroll
  for (int u = 0; u < PER; ++u)
    if (first[u]) uniq[rank++] = key[threadIdx.x * PER + u];
  __syncthreads();
  int* out = nodes + e0 * NPE;
  for (int l = threadIdx.x; l < total; l += kBlock) out[l] = uniq[l] | ((int)(fm[uniq[l]] & 7) << 28);
  for (int i = threadIdx.x; i < refs; i += kBlock) {
    const int id = src[i];
    int lo = 0, hi = total - 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (uniq[mid] < id) lo = mid + 1;
      else hi = mid;
    }
    loc[e0 * NPE + i] = (uint16_t)lo;
  }
}

// Bounds on the absolute row sums of a quadratic tet's K and M, added per node: with d_i = grad N_i at the four
// Gauss points, sum_j sum_l |K_ik,jl| <= V/4 sum_q (lambda |d_ik| sum_j |d_j|_1 + mu |d_i|_1 sum_j |d_jk| + mu sum_j
// |d_i . d_j|) (the absolute values inside the sum over the points: at most a bit looser than outside).
__global__ void __launch_bounds__(kBlock) k_abs_rows10(int64_t E, const int32_t* __restrict__ conn,
                                                       const float* __restrict__ rec, float* __restrict__ mrow,
                                                       float* __restrict__ krow) {
  const float GA = 0.5854101966249685f, GB = 0.1381966011250105f;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < E; e += (int64_t)gridDim.x * blockDim.x) {
    float r[12];
    load_rec(rec + e * kRec, r);
    float g[4][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      g[1][k] = r[k], g[2][k] = r[3 + k], g[3][k] = r[6 + k];
      g[0][k] = -(g[1][k] + g[2][k] + g[3][k]);
    }
    const float lam = r[9] * 0.25f, mu = r[10] * 0.25f, rv = r[11] * 20.0f;
    float row[10][3] = {};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float d[10][3], s1 = 0.f, sk[3] = {0.f, 0.f, 0.f};
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          d[a][k] = (4.0f * (a == q ? GA : GB) - 1.0f) * g[a][k];
#pragma unroll
          for (int b = a + 1; b < 4; ++b)
            d[edge_node10(a, b)][k] = 4.0f * ((a == q ? GA : GB) * g[b][k] + (b == q ? GA : GB) * g[a][k]);
        }
#pragma unroll
      for (int i = 0; i < 10; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) sk[k] += fabsf(d[i][k]);
      s1 = sk[0] + sk[1] + sk[2];
#pragma unroll
      for (int i = 0; i < 10; ++i) {
        float dd = 0.f;
#pragma unroll
        for (int j = 0; j < 10; ++j) dd += fabsf(d[i][0] * d[j][0] + d[i][1] * d[j][1] + d[i][2] * d[j][2]);
        const float n1 = fabsf(d[i][0]) + fabsf(d[i][1]) + fabsf(d[i][2]);
#pragma unroll
        for (int k = 0; k < 3; ++k) row[i][k] += lam * fabsf(d[i][k]) * s1 + mu * (n1 * sk[k] + dd);
      }
    }
#pragma unroll
    for (int i = 0; i < 10; ++i) {
      const int64_t n = conn[e * 10 + i];
#pragma unroll
      for (int k = 0; k < 3; ++k) atomicAdd(krow + n * 3 + k, row[i][k]);
      // sum_j |m_ij|: corner (6 + 3 + 3 x 4 + 3 x 6) / 420, edge (2 x 4 + 2 x 6 + 32 + 4 x 16 + 8) / 420
      atomicAdd(mrow + n, rv * ((i < 4 ? 39.0f : 124.0f) / 420.0f));
    }
  }
}

// Shared memory: the per-case |p| maxima (one set a tile parity), a row a node of the tile with its p (3 R values)
// and its fixed-point sums (3 R), and two buffers of the tile's tables (node list, element records, local indices),
// the next tile's copied while this one is applied.  A row is padded so that the groups of R lanes that read the
// rows of different elements' nodes spread over the banks (R values mod 32).
__host__ __device__ constexpr int tile_row(int r) { return 6 * r + (r < 32 ? r : 0); }
struct TileLayout {
  size_t row, node, rec, loc, node_sz, rec_sz, loc_sz, total;
};
__host__ __device__ inline TileLayout tile_layout(int npe, int nloc, int per_tile, int rpad) {
  auto up = [](size_t x) { return (x + 15) & ~(size_t)15; };
  TileLayout L;
  L.node_sz = up(sizeof(int) * (size_t)nloc), L.rec_sz = sizeof(float) * kRec * per_tile, L.loc_sz = up((size_t)2 * npe * per_tile);
  L.row = 256;
  L.node = L.row + (size_t)nloc * tile_row(rpad) * 4;
  L.rec = L.node + 2 * L.node_sz;
  L.loc = L.rec + 2 * L.rec_sz;
  L.total = L.loc + 2 * L.loc_sz;
  return L;
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// A tile's elements of cases c .. added to q in FP32 (a tile whose fixed-point bound is not finite).
template <int NPE, bool DOT>
__device__ __noinline__ float tile_direct(const ElemTiles& et, int64_t e0, int items, int rpad, int c,
                                         const float* rec, const float* p, float* q, const int* snode, float aM,
                                         float aK) {
  const int per_node = 3 * rpad;
  float td = 0.f;
  for (int it = threadIdx.x; it < items; it += kBlock) {
    const int64_t e = e0 + it / rpad;
    float r[12];
    load_rec(rec + e * kRec, r);
    int nd[NPE];
#pragma unroll
    for (int a = 0; a < NPE; ++a) nd[a] = snode[et.loc[e * NPE + a]];
    auto ld = [&](int a, float (&P)[3]) {
#pragma unroll
      for (int k = 0; k < 3; ++k)
        P[k] = p[(int64_t)(nd[a] & 0x0fffffff) * per_node + k * rpad + c];
    };
    auto fl = [&](int a, const float (&Q)[3]) {
#pragma unroll
      for (int k = 0; k < 3; ++k)
        if (dof_free((uint8_t)((nd[a] >> 28) & 7), k))
          atomicAdd(q + (int64_t)(nd[a] & 0x0fffffff) * per_node + k * rpad + c, Q[k]);
    };
    if constexpr (NPE == 4) elem4<DOT, false, float, float>(ld, ld, fl, r, aM, aK, td);
    else elem10<DOT, float, float>(ld, fl, r, aM, aK, td);
  }
  return td;
}

// R cases, one a thread.  A thread's case is fixed (the block is a multiple of R), so its scale is one register a
// tile, and with R a constant the offsets of a node's values are immediates.  Both element types are bound by
// instruction issue and shared-memory latency (quadratic: 1077 instructions an element and case, 737 of them FP32
// arithmetic, 0.68 a clock and scheduler).  386,370 linear tets, 8 cases: 57.8 us by global atomics, 52 without the
// staged tables, 43 with pairs of cases a thread (their atomics use every other bank), 41 so; 128 elements a tile
// 45, 64 55.  786,432 quadratic tets, 16 cases: 621 -> 529 us (pairs of cases at 8 warps an SM: 685).
template <int NPE, int R, bool DOT>
__global__ void __launch_bounds__(kBlock, NPE == 4 ? 4 : 2) k_elem_tile(ElemTiles et, int64_t E, const float* __restrict__ rec,
                                                         const float* __restrict__ p, float* __restrict__ q, float aM,
                                                         float aK, Reducer red, CgCase* sc, double* ptq_out,
                                                         const int* gate) {
  if (gate && *gate == 0) return;
  extern __shared__ __align__(16) unsigned char smem[];
  const TileLayout L = tile_layout(NPE, et.nloc_max, et.per_tile, R);
  constexpr int ROW = tile_row(R), F4 = 3 * R / 4;   // a node's row, its 16-byte pieces
  float* rows = reinterpret_cast<float*>(smem + L.row);
  const int c = threadIdx.x & (R - 1), c4 = (threadIdx.x << 2) & (R - 1);
  const float bco = fabsf(aM) * et.abs_m + fabsf(aK) * et.abs_k;
  // tables of tile t into buffer b: 16-byte pieces (the arrays are padded to them)
  auto stage = [&](int t, int b, int nl) {
    const int64_t e0 = (int64_t)t * et.per_tile;
    const int ne = (int)min((int64_t)et.per_tile, E - e0);
    const unsigned char* gn = reinterpret_cast<const unsigned char*>(et.nodes + e0 * NPE);
    const unsigned char* gr = reinterpret_cast<const unsigned char*>(rec + e0 * kRec);
    const unsigned char* gl = reinterpret_cast<const unsigned char*>(et.loc + e0 * NPE);
    for (int i = threadIdx.x * 16; i < nl * 4; i += kBlock * 16) cp_async16(smem + L.node + b * L.node_sz + i, gn + i);
    for (int i = threadIdx.x * 16; i < ne * kRec * 4; i += kBlock * 16) cp_async16(smem + L.rec + b * L.rec_sz + i, gr + i);
    for (int i = threadIdx.x * 16; i < ne * NPE * 2; i += kBlock * 16) cp_async16(smem + L.loc + b * L.loc_sz + i, gl + i);
  };
  auto field = [&](int m) { return (int)((__float_as_uint(bco * __int_as_float(m)) >> 23) & 0xffu); };
  auto expo = [](int f) { return max(f - 126, -96); };               // bound < 2^expo (fixed_expo)
  double dot = 0.0;
  int* spm0 = reinterpret_cast<int*>(smem);
  if (threadIdx.x < 64) spm0[threadIdx.x] = 0;
  int nl = (int)blockIdx.x < et.n_tiles ? et.count[blockIdx.x] : 0;
  if (nl) stage(blockIdx.x, 0, nl);
  cp_commit();
  int b = 0;
  for (int t = blockIdx.x; t < et.n_tiles; t += gridDim.x, b ^= 1) {
    const int tn = t + gridDim.x;
    const int nl_next = tn < et.n_tiles ? et.count[tn] : 0;
    const int* snode = reinterpret_cast<const int*>(smem + L.node + b * L.node_sz);
    int* spm = spm0 + 32 * b;
    const int64_t e0 = (int64_t)t * et.per_tile;
    const int ne = (int)min((int64_t)et.per_tile, E - e0);
    cp_wait<0>();
    __syncthreads();
    for (int i = threadIdx.x; i < nl * F4; i += kBlock) {
      const int l = i / F4, j = 4 * (i - l * F4);
      float* row = rows + l * ROW;
      cp_async16(row + j, p + (int64_t)(snode[l] & 0x0fffffff) * (3 * R) + j);
      *reinterpret_cast<int4*>(row + 3 * R + j) = make_int4(0, 0, 0, 0);
    }
    cp_commit();
    if (nl_next) stage(tn, b ^ 1, nl_next);
    cp_commit();
    cp_wait<1>();      // (this thread's own pieces, whose maxima it takes; a piece's four cases are c4 .. c4 + 3)
    int m4[4] = {0, 0, 0, 0};
    for (int i = threadIdx.x; i < nl * F4; i += kBlock) {
      const int l = i / F4;
      const int4 v = *reinterpret_cast<const int4*>(rows + l * ROW + 4 * (i - l * F4));   // (the bit patterns of |v| are ordered, NaN above infinity)
      m4[0] = max(m4[0], v.x & 0x7fffffff), m4[1] = max(m4[1], v.y & 0x7fffffff);
      m4[2] = max(m4[2], v.z & 0x7fffffff), m4[3] = max(m4[3], v.w & 0x7fffffff);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      for (int o = 16; o >= R / 4; o >>= 1) m4[u] = max(m4[u], __shfl_xor_sync(0xffffffffu, m4[u], o));
      if ((int)(threadIdx.x & 31) < R / 4) atomicMax(spm + c4 + u, m4[u]);
    }
    __syncthreads();
    const int fc = field(spm[c]);
    const float scale = pow2(30 - expo(fc));
    const bool direct = fc == 0xff;
    float td = 0.f;
    if (direct) {
      td = tile_direct<NPE, DOT>(et, e0, ne * R, R, c, rec, p, q, snode, aM, aK);
    } else {
      const float* srec = reinterpret_cast<const float*>(smem + L.rec + b * L.rec_sz);
      const uint32_t* sloc = reinterpret_cast<const uint32_t*>(smem + L.loc + b * L.loc_sz);
      for (int it = threadIdx.x; it < ne * R; it += kBlock) {
        const int el = it / R;
        float r[12];
        const float4* r4 = reinterpret_cast<const float4*>(srec + el * kRec);
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const float4 v = r4[u];
          r[4 * u] = v.x, r[4 * u + 1] = v.y, r[4 * u + 2] = v.z, r[4 * u + 3] = v.w;
        }
        float* o[NPE];
#pragma unroll
        for (int a = 0; a < NPE / 2; ++a) {
          const uint32_t w = sloc[el * (NPE / 2) + a];
          o[2 * a] = rows + (w & 0xffff) * ROW + c;
          o[2 * a + 1] = rows + (w >> 16) * ROW + c;
        }
        auto ld = [&](int a, float (&P)[3]) {
#pragma unroll
          for (int k = 0; k < 3; ++k) P[k] = o[a][k * R];
        };
        auto fl = [&](int a, const float (&Q)[3]) {
#pragma unroll
          for (int k = 0; k < 3; ++k) atomicAdd(reinterpret_cast<int*>(o[a] + (3 + k) * R), __float2int_rn(Q[k] * scale));
        };
        if constexpr (NPE == 4) elem4<DOT, false, float, float>(ld, ld, fl, r, aM, aK, td);
        else elem10<DOT, float, float>(ld, fl, r, aM, aK, td);
      }
    }
    if constexpr (DOT) dot += (double)td;
    __syncthreads();
    const float w4[4] = {pow2(expo(field(spm[c4])) - 30), pow2(expo(field(spm[c4 + 1])) - 30),
                         pow2(expo(field(spm[c4 + 2])) - 30), pow2(expo(field(spm[c4 + 3])) - 30)};
    if (threadIdx.x < 32) spm0[32 * (b ^ 1) + threadIdx.x] = 0;     // (the next tile's; its last readers are a barrier back)
    for (int i = threadIdx.x; i < nl * F4; i += kBlock) {
      const int l = i / F4, raw = snode[l], j = 4 * (i - l * F4);
      if (!dof_free((uint8_t)((raw >> 28) & 7), j / R)) continue;
      const int4 v = *reinterpret_cast<const int4*>(rows + l * ROW + 3 * R + j);
      atomicAdd(reinterpret_cast<float4*>(q + (int64_t)(raw & 0x0fffffff) * (3 * R) + j),
                make_float4((float)v.x * w4[0], (float)v.y * w4[1], (float)v.z * w4[2], (float)v.w * w4[3]));
    }
    nl = nl_next;
  }
  if constexpr (DOT) {
    double v[1] = {dot};
    if (block_reduce_last<1>(v, R, red)) ebe_tail(red, sc, ptq_out, R);
  }
}

}  // namespace

void free_elem_tiles(ElemTiles* t) {
  cudaFree(const_cast<int*>(t->count));
  cudaFree(const_cast<int*>(t->nodes));
  cudaFree(const_cast<uint16_t*>(t->loc));
  *t = ElemTiles{};
}

cudaError_t build_elem_tiles(int npe, int64_t E, int64_t N, const int32_t* conn, const uint8_t* fm, const float* rec32,
                             ElemTiles* out, cudaStream_t s) {
  *out = ElemTiles{};
  // elements a tile (at most kSortMax references): linear 256, quadratic 48
  const int per = npe == 4 ? 256 : 48;
  const int64_t tiles = (E + per - 1) / per;
  if (N >= ((int64_t)1 << 28) || tiles < 2 * sm_count()) return cudaSuccess;
  int *count = nullptr, *nodes = nullptr;
  uint16_t* loc = nullptr;
  float* rows = nullptr;       // [3 N] K rows, [N] M rows, their maxima (2), the counts' statistics (2 x 8 bytes)
  struct {
    float mk, mm;
    unsigned long long nmax, sum;
  } h{};
  const int64_t tail = ((4 * N + 1) & ~(int64_t)1);
  cudaError_t e = cudaMalloc(&count, sizeof(int) * tiles);
  if (e == cudaSuccess) e = cudaMalloc(&nodes, sizeof(int) * npe * E + 16);
  if (e == cudaSuccess) e = cudaMalloc(&loc, sizeof(uint16_t) * npe * E + 16);
  if (e == cudaSuccess) e = cudaMalloc(&rows, sizeof(float) * tail + sizeof(h));
  if (e == cudaSuccess) e = cudaMemsetAsync(rows, 0, sizeof(float) * tail + sizeof(h), s);
  if (e == cudaSuccess) {
    int* mx = reinterpret_cast<int*>(rows + tail);
    unsigned long long* stats = reinterpret_cast<unsigned long long*>(rows + tail + 2);
    if (npe == 4) {
      k_tile_nodes<4><<<(unsigned)tiles, kBlock, 0, s>>>(E, per, conn, fm, count, nodes, loc, stats);
      e = launch_abs_rows4(E, reinterpret_cast<const int4*>(conn), rec32, rows + 3 * N, rows, s);
    } else {
      k_tile_nodes<10><<<(unsigned)tiles, kBlock, 0, s>>>(E, per, conn, fm, count, nodes, loc, stats);
      k_abs_rows10<<<grid_for(E), kBlock, 0, s>>>(E, conn, rec32, rows + 3 * N, rows);
    }
    if (e == cudaSuccess) e = launch_max_abs(3 * N, rows, mx, s);
    if (e == cudaSuccess) e = launch_max_abs(N, rows + 3 * N, mx + 1, s);
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, rows + tail, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(rows);
  // worth it where a tile's nodes are shared by at least three of its elements on average
  if (e != cudaSuccess || (double)h.sum * 3.0 > (double)E * npe) {
    cudaFree(count);
    cudaFree(nodes);
    cudaFree(loc);
    return e;
  }
  out->n_tiles = (int)tiles, out->per_tile = per, out->nloc_max = (int)h.nmax;
  out->count = count, out->nodes = nodes, out->loc = loc;
  out->abs_m = h.mm * 1.01f, out->abs_k = h.mk * 1.01f;    // (1%: the FP32 rounding of the bounds and products)
  return cudaSuccess;
}

bool elem_tile_fits(int npe, const ElemTiles& et, int rpad, const void* p, const void* q) {
  // two blocks an SM; 16-byte pieces of four cases.  Quadratic tets from 8 cases on: with 4 the tiles' passes over
  // the nodes weigh more than the atomics they save (786,432 tets: 244 us against 184 for the plain kernel).
  return et.n_tiles > 0 && rpad >= (npe == 4 ? 4 : 8) &&
         tile_layout(npe, et.nloc_max, et.per_tile, rpad).total <= 110 * 1024 &&
         ((reinterpret_cast<uintptr_t>(p) | reinterpret_cast<uintptr_t>(q)) & 15) == 0;
}

template <int NPE>
static cudaError_t launch_tile_t(const ElemTiles& et, int64_t E, int rpad, const float* rec32, const float* p, float* q,
                                 double aM, double aK, const Reducer* red, CgCase* sc, double* ptq, const int* gate,
                                 cudaStream_t s) {
  const size_t smem = tile_layout(NPE, et.nloc_max, et.per_tile, rpad).total;
  const Reducer rd = red ? *red : Reducer{nullptr, nullptr, nullptr};
  auto run = [&](auto kfn) {
    int per_sm = 1;
    cudaError_t e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kfn, kBlock, smem);
    if (e != cudaSuccess) return e;
    int grid = sm_count() * (per_sm < 1 ? 1 : per_sm);
    if (grid > et.n_tiles) grid = et.n_tiles;
    if (grid > red_grid_cap()) grid = red_grid_cap();
    kfn<<<grid, kBlock, smem, s>>>(et, E, rec32, p, q, (float)aM, (float)aK, rd, red ? sc : nullptr, red ? ptq : nullptr,
                                   gate);
    return cudaGetLastError();
  };
  auto by_dot = [&](auto r) {
    constexpr int R = decltype(r)::value;
    if constexpr (NPE == 10) {
      if (red) return run(k_elem_tile<NPE, R, true>);
    }
    return run(k_elem_tile<NPE, R, false>);
  };
  switch (rpad) {
    case 4: return by_dot(std::integral_constant<int, 4>{});
    case 8: return by_dot(std::integral_constant<int, 8>{});
    case 16: return by_dot(std::integral_constant<int, 16>{});
    default: return by_dot(std::integral_constant<int, 32>{});
  }
}

// q must be zero; Dirichlet rows stay zero.
cudaError_t launch_elem_tile(int npe, const ElemTiles& et, int64_t E, int rpad, const float* rec32, const float* p,
                             float* q, double aM, double aK, const Reducer* red, CgCase* sc, double* ptq,
                             const int* gate, cudaStream_t s) {
  if (npe == 4) return launch_tile_t<4>(et, E, rpad, rec32, p, q, aM, aK, nullptr, nullptr, nullptr, gate, s);
  return launch_tile_t<10>(et, E, rpad, rec32, p, q, aM, aK, red, sc, ptq, gate, s);
}

}  // namespace fem
