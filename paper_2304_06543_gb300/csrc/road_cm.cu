// Cost matrix from a road network (Section 3.4 "Demand-service cost matrix
// construction"; Section 5: the paper's CM is the shortest road distance from
// every demand node to every service center of the New Delhi network).
//
// One CTA per center computes single-source shortest paths over the CSR graph
// by label correcting in near and far steps (the bucket idea of
// delta-stepping, Meyer and Sanders 2003, with two buckets): a step relaxes
// the edges of the nodes whose label dropped below the current threshold in
// the step before; a node whose label dropped but is not below it waits in
// the far list; when no near node is left the threshold moves up and the far
// list is split again.  Labels only decrease and lengths are positive integers,
// so the sweeps end with the exact shortest distances whatever order the
// relaxations take; the CM is therefore bit-identical to a sequential
// Dijkstra.  The labels of all centers (k x V int32) stay L2-resident for
// road graphs of the paper's size (65,000 nodes, about 100 centers).
// A gather then writes CM[d][s] = dist_s(demand[d]), demand-major.
#include <algorithm>
#include <cstdint>
#include <cstring>

#include "lbdd_internal.h"

namespace lbdd {

constexpr int kRoadThreads = 512;
constexpr int32_t kRoadInf = INT32_MAX;

// err[0]: bad graph or ids; err[1]: largest length; err[2]: unreachable
// demand; err[3]: step limit reached (cannot happen with positive lengths);
// err[4..5]: sum of all lengths (64 bits); err[6]: number of roads.
__global__ void road_check(int32_t V, const int32_t* __restrict__ row_ptr,
                           const int32_t* __restrict__ col, const int32_t* __restrict__ w,
                           int32_t k, const int32_t* __restrict__ centers, int32_t n,
                           const int32_t* __restrict__ demand, int* err) {
  const int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t gs = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v = g; v < V; v += gs)
    if (row_ptr[v] > row_ptr[v + 1] || row_ptr[v] < 0) atomicExch(err, 1);
  const int32_t E = row_ptr[V];
  if (row_ptr[0] != 0 || E < 0) atomicExch(err, 1);
  if (g == 0) err[6] = E;
  int mx = 0;
  unsigned long long sum = 0;
  for (int64_t e = g; e < E; e += gs) {
    const int32_t we = w[e];
    if (we < 1 || (uint32_t)col[e] >= (uint32_t)V) atomicExch(err, 1);
    mx = max(mx, we);
    sum += (unsigned long long)max(we, 0);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  for (int off = 16; off > 0; off >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, off);
  if ((threadIdx.x & 31) == 0 && mx > 0) {
    atomicMax(err + 1, mx);
    atomicAdd(reinterpret_cast<unsigned long long*>(err + 4), sum);
  }
  for (int64_t s = g; s < k; s += gs)
    if ((uint32_t)centers[s] >= (uint32_t)V) atomicExch(err, 1);
  for (int64_t d = g; d < n; d += gs)
    if ((uint32_t)demand[d] >= (uint32_t)V) atomicExch(err, 1);
}

// The graph as the steps read it: 8 (neighbour, length) pairs per node, absent
// ones marked -1, so that a node's edges are one 64-byte read that depends on
// nothing but the node.  A node of more than 8 roads keeps 7 and points to the
// rest of its CSR row: (-2, first remaining edge).
constexpr int kRoadDeg = 8;

__global__ void road_pack(int32_t V, const int32_t* __restrict__ row_ptr,
                          const int32_t* __restrict__ col, const int32_t* __restrict__ w,
                          int2* __restrict__ adj) {
  const int64_t total = (int64_t)V * kRoadDeg;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = (int32_t)(i / kRoadDeg), q = (int32_t)(i % kRoadDeg);
    const int32_t e0 = row_ptr[v], deg = row_ptr[v + 1] - e0;
    int2 a = make_int2(-1, 0);
    if (q == kRoadDeg - 1 && deg > kRoadDeg) a = make_int2(-2, e0 + q);
    else if (q < deg) a = make_int2(col[e0 + q], w[e0 + q]);
    adj[i] = a;
  }
}

// Shared memory of a CTA: three bitmaps (one bit per node: in the near list
// being read, in the one being written, in the far list; in global memory for
// graphs past kRoadSmemNodes) and the first kRoadQueue entries of each of
// three lists (the rest spill to global memory).
constexpr int kRoadQueue = 4096;
constexpr int32_t kRoadSmemNodes = 400000;

__host__ __device__ inline size_t road_bitmap_words(int32_t V) { return ((size_t)V + 31) / 32; }
static size_t road_smem_bytes(int32_t V) {
  return 12 * (size_t)kRoadQueue + (V <= kRoadSmemNodes ? 12 * road_bitmap_words(V) : 0);
}

// Sets `bit` of a bitmap word where `on`; returns the word as it was (all ones
// where not).  Predicated instead of branched around, so that the atomics of
// a node's edges are in flight together.
template <bool SMEM>
__device__ __forceinline__ uint32_t mark_if(bool on, uint32_t* word, uint32_t bit) {
  uint32_t old;
  if constexpr (SMEM)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.u32 %0, 0xffffffff;\n\t"
        "@p atom.shared.or.b32 %0, [%1], %2;\n\t}"
        : "=r"(old) : "r"(smem_u32(word)), "r"(bit), "r"((uint32_t)on) : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\tmov.u32 %0, 0xffffffff;\n\t"
        "@p atom.global.or.b32 %0, [%1], %2;\n\t}"
        : "=r"(old) : "l"(word), "r"(bit), "r"((uint32_t)on) : "memory");
  return old;
}
__device__ __forceinline__ void lower_if(bool on, int32_t* label, int32_t v) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.global.min.s32 [%0], %1;\n\t}"
               ::"l"(label), "r"(v), "r"((uint32_t)on) : "memory");
}

// A step is a chain of memory latencies (node, its label and row, edges,
// neighbour labels), so there should be few steps and little in each: the
// threshold keeps a node from being relaxed again for every detour that
// reaches it first (65,536 nodes in a grid: 1.1 relaxations per node instead
// of up to 12, in about as many steps).  The lists and the marks live in
// shared memory, a thread has eight edges of a node in flight together, and a
// label is lowered by a reduction that returns nothing (the label read before
// decides whether the neighbour is listed; one that was lowered further in
// between is listed all the same).  65,536 nodes, 109 centers: 6.6 ms per
// call with one list and marks in global memory, 1.74 ms now.  (Marks spread over
// banks, and one atomic per warp instead of one per node for a list's length,
// measured no faster: what a step issues counts for more than its conflicts.)
template <bool SMEM>
__global__ void __launch_bounds__(kRoadThreads)
road_sssp(int32_t V, const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ col,
          const int32_t* __restrict__ w, const int2* __restrict__ adj, int32_t k,
          const int32_t* __restrict__ centers, int32_t delta, int32_t* dist, int32_t* queues, uint32_t* marks, int* err) {
  constexpr int U = kRoadDeg;
  extern __shared__ __align__(16) uint32_t road_smem[];
  __shared__ int s_near[3], s_far[2], s_min;
  const int tid = threadIdx.x, lane = tid & 31;
  const size_t words = road_bitmap_words(V);
  int32_t* sq = reinterpret_cast<int32_t*>(road_smem);            // [3][kRoadQueue]
  uint32_t* bits = SMEM ? road_smem + 3 * kRoadQueue : marks + 3 * words * blockIdx.x;   // [3][words]
  uint32_t* far_bits = bits + 2 * words;
  int32_t* gq = queues + (int64_t)blockIdx.x * 3 * V;             // [3][V]
  auto item = [&](int list, int i) {
    return i < kRoadQueue ? sq[list * kRoadQueue + i] : gq[(int64_t)list * V + i];
  };
  auto put = [&](int list, int at, int32_t v) {
    if (at < kRoadQueue) sq[list * kRoadQueue + at] = v;
    else gq[(int64_t)list * V + at] = v;
  };
  // appends v to a list; the lanes that are together share one atomic
  auto append = [&](int list, int* cnt, int32_t v, bool push) {
    const unsigned act = __activemask();
    const unsigned who = __ballot_sync(act, push);
    if (who == 0) return;
    const int leader = __ffs(who) - 1;
    int at = 0;
    if (lane == leader) at = atomicAdd(cnt, __popc(who));
    at = __shfl_sync(act, at, leader) + __popc(who & ((1u << lane) - 1u));
    if (push) put(list, at, v);
  };
  for (int32_t s = blockIdx.x; s < k; s += gridDim.x) {
    int32_t* d = dist + (int64_t)s * V;
    for (int32_t v = tid; v < V; v += kRoadThreads) d[v] = kRoadInf;
    for (size_t i = tid; i < 3 * words; i += kRoadThreads) bits[i] = 0;
    __syncthreads();
    if (tid == 0) {
      d[centers[s]] = 0;
      sq[0] = centers[s];
      s_near[0] = s_near[1] = s_near[2] = 0;
      s_far[0] = s_far[1] = 0;
    }
    __syncthreads();
    int ln = 0, lx = 1, lf = 2;       // lists: near being read, near being written, far
    int na = 1, par = 0, fpar = 0, c3 = 1;
    int64_t T = delta;                // near: labels below T
    bool ok = true;
    for (int64_t step = 0; ok; ++step) {
      if (step > 4 * (int64_t)V) {    // positive lengths: at most V near steps and V splits
        ok = false;
        break;
      }
      if (na == 0) {
        // split the far list: both near lists are empty
        const int nf = s_far[fpar];
        if (nf == 0) break;
        __syncthreads();              // nf read by all
        if (tid == 0) {
          s_far[fpar ^ 1] = 0;
          s_near[0] = s_near[1] = s_near[2] = 0;
          s_min = kRoadInf;
        }
        __syncthreads();
        int mn = kRoadInf;
        for (int i = tid; i < nf; i += kRoadThreads) {
          const int32_t u = item(lf, i);
          const int32_t du = __ldcg(d + u);
          const bool keep = du >= T + delta, near = du >= T && !keep;   // below T: relaxed already
          if (!keep) atomicAnd(far_bits + (u >> 5), ~(1u << (u & 31)));
          else mn = min(mn, du);
          append(ln, &s_near[0], u, near);
          append(lx, &s_far[fpar ^ 1], u, keep);
        }
        if (mn != kRoadInf) atomicMin(&s_min, mn);
        __syncthreads();
        na = s_near[0];
        c3 = 1;
        fpar ^= 1;
        const int t = lx;             // the kept nodes are the far list now
        lx = lf;
        lf = t;
        T = na == 0 && s_far[fpar] > 0 ? (int64_t)s_min : T + delta;
        __syncthreads();              // s_min read by all
        continue;
      }
      uint32_t* bin = bits + par * words;
      uint32_t* bout = bits + (par ^ 1) * words;
      const int c3n = c3 == 2 ? 0 : c3 + 1;
      if (tid == 0) s_near[c3n] = 0;
      for (int i = tid; i < na; i += kRoadThreads) {
        const int32_t u = item(ln, i);
        const int4* row = reinterpret_cast<const int4*>(adj + (int64_t)u * kRoadDeg);
        // sums and labels as unsigned words: a label is a simple path's length
        // (below 2^31, checked by the host), one road more may reach 2^32 - 1
        int32_t v[U];
        uint32_t nd[U], dv[U];
#pragma unroll
        for (int q = 0; q < U; q += 2) {
          const int4 x = __ldg(row + q / 2);
          v[q] = x.x;
          nd[q] = x.y;
          v[q + 1] = x.z;
          nd[q + 1] = x.w;
        }
        const int32_t du = __ldcg(d + u);
        bin[u >> 5] = 0;   // every set bit of this map is in the list being read
        int32_t rest = 0, end = 0;
        if (v[U - 1] == -2) {
          rest = (int32_t)nd[U - 1];
          end = __ldg(row_ptr + u + 1);
        }
        for (;;) {
#pragma unroll
          for (int q = 0; q < U; ++q) dv[q] = v[q] >= 0 ? (uint32_t)__ldcg(d + v[q]) : 0u;
          uint32_t old[U];
#pragma unroll
          for (int q = 0; q < U; ++q) {
            nd[q] += (uint32_t)du;
            const bool on = nd[q] < dv[q];
            const int32_t x = on ? v[q] : 0;
            lower_if(on, d + x, (int32_t)nd[q]);
            old[q] = mark_if<SMEM>(on, (nd[q] < T ? bout : far_bits) + (x >> 5), 1u << (x & 31));
          }
          unsigned near = 0, far = 0;
#pragma unroll
          for (int q = 0; q < U; ++q) {
            if (!(old[q] >> (v[q] & 31) & 1)) {   // all ones where nothing was lowered
              if (nd[q] < T) near |= 1u << q;
              else far |= 1u << q;
            }
          }
          int an = near ? atomicAdd(&s_near[c3], __popc(near)) : 0;
          int af = far ? atomicAdd(&s_far[fpar], __popc(far)) : 0;
#pragma unroll
          for (int q = 0; q < U; ++q) {
            if (near >> q & 1) put(lx, an++, v[q]);
            if (far >> q & 1) put(lf, af++, v[q]);
          }
          if (rest >= end) break;
#pragma unroll
          for (int q = 0; q < U; ++q) {
            const bool on = rest + q < end;
            v[q] = on ? __ldg(col + rest + q) : -1;
            nd[q] = on ? (uint32_t)__ldg(w + rest + q) : 0u;
          }
          rest += U;
        }
      }
      __syncthreads();
      na = s_near[c3];
      c3 = c3n;
      par ^= 1;
      const int t = ln;
      ln = lx;
      lx = t;
    }
    if (!ok && tid == 0) atomicExch(err + 3, 1);
    __syncthreads();
  }
}

// CM[dd][s] = dist_s(demand[dd]), 32 x 32 entries at a time through shared
// memory: the labels are read along a center's row (demand nodes are mostly
// in order), CM is written along its rows.
__global__ void __launch_bounds__(256)
road_gather(int32_t V, int32_t k, int32_t n, const int32_t* __restrict__ dist,
            const int32_t* __restrict__ demand, int32_t* cm, int64_t ld, int* err) {
  __shared__ int32_t tile[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t ks = (k + 31) / 32;
  const int64_t tiles = (int64_t)((n + 31) / 32) * ks;
  bool bad = false;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const int32_t d0 = (int32_t)(t / ks) * 32, s0 = (int32_t)(t % ks) * 32;
    const int32_t node = d0 + lane < n ? __ldg(demand + d0 + lane) : -1;
    for (int i = warp; i < 32; i += 8) {
      int32_t v = 1;
      if (node >= 0 && s0 + i < k) {
        v = __ldcg(dist + (int64_t)(s0 + i) * V + node);
        bad |= v == kRoadInf || v < 1;
      }
      tile[i][lane] = v;
    }
    __syncthreads();
    for (int i = warp; i < 32; i += 8)
      if (d0 + i < n && s0 + lane < k) cm[(int64_t)(d0 + i) * ld + s0 + lane] = tile[lane][i];
    __syncthreads();
  }
  if (bad) atomicExch(err + 2, 1);
}

}  // namespace lbdd

using namespace lbdd;

extern "C" int lbdd_road_cm(int32_t V, const int32_t* row_ptr, const int32_t* col,
                            const int32_t* w, int32_t k, const int32_t* centers, int32_t n,
                            const int32_t* demand, int32_t* cm, int64_t ld, void* stream) {
  if (V < 1 || k < 1 || n < 1 || ld < k || !row_ptr || !col || !w || !centers || !demand || !cm)
    return LBDD_ERR_ARG;
  int dev = 0, sms = 0;
  int rc = check_device(&dev, &sms);
  if (rc) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int grid = std::min(k, sms);
  unsigned char* base = nullptr;
  int* err = nullptr;
  auto release = [&]() {
    if (base) cudaFreeAsync(base, st);
    cudaFreeAsync(err, st);
    cudaStreamSynchronize(st);
  };
  cudaError_t e = cudaMallocAsync(reinterpret_cast<void**>(&err), 8 * sizeof(int), st);
  if (!e) e = cudaMemsetAsync(err, 0, 8 * sizeof(int), st);
  if (!e) {
    road_check<<<sms * 4, 256, 0, st>>>(V, row_ptr, col, w, k, centers, n, demand, err);
    e = cudaGetLastError();
  }
  int h[8] = {};
  if (!e) e = cudaMemcpyAsync(h, err, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (!e) e = cudaStreamSynchronize(st);
  if (e) { rc = cuda_fail(e, "lbdd_road_cm check"); release(); return rc; }
  // labels are int32: every path length must fit
  if (h[0] != 0 || (int64_t)h[1] * (V - 1) >= (int64_t)kRoadInf) { release(); return LBDD_ERR_ARG; }
  // one allocation for all scratch
  auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t o_queues = al(4ull * k * V), o_adj = o_queues + al(12ull * grid * V);
  const size_t o_marks = o_adj + al(sizeof(int2) * kRoadDeg * (size_t)V);
  const size_t o_end = o_marks + (V > kRoadSmemNodes ? 12ull * grid * road_bitmap_words(V) : 0);
  e = cudaMallocAsync(reinterpret_cast<void**>(&base), o_end, st);
  int32_t* dist = reinterpret_cast<int32_t*>(base);
  int32_t* queues = reinterpret_cast<int32_t*>(base + o_queues);
  int2* adj = reinterpret_cast<int2*>(base + o_adj);
  uint32_t* marks = reinterpret_cast<uint32_t*>(base + o_marks);   // bitmaps past shared memory
  const size_t smem = road_smem_bytes(V);
  // threshold step: four mean lengths (1.05 to 1.1 relaxations per node on
  // grids; half as much takes a fifth more steps, twice as much 1.2
  // relaxations)
  uint64_t sum = 0;
  std::memcpy(&sum, h + 4, sizeof(sum));
  const uint64_t roads = (uint64_t)std::max(1, h[6]);
  const int32_t delta = (int32_t)std::min<uint64_t>(1u << 30, std::max<uint64_t>(1, 4 * sum / roads));
  auto sssp = V <= kRoadSmemNodes ? road_sssp<true> : road_sssp<false>;
  if (!e)   // the largest any graph asks for
    e = cudaFuncSetAttribute(sssp, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)road_smem_bytes(kRoadSmemNodes));
  if (!e) {
    road_pack<<<sms * 8, 256, 0, st>>>(V, row_ptr, col, w, adj);
    sssp<<<grid, kRoadThreads, smem, st>>>(V, row_ptr, col, w, adj, k, centers, delta, dist, queues,
                                           marks, err);
    e = cudaGetLastError();
  }
  if (!e) {
    road_gather<<<sms * 8, 256, 0, st>>>(V, k, n, dist, demand, cm, ld, err);
    e = cudaGetLastError();
  }
  if (!e) e = cudaMemcpyAsync(h, err, sizeof(h), cudaMemcpyDeviceToHost, st);
  if (!e) e = cudaStreamSynchronize(st);
  if (e) { rc = cuda_fail(e, "lbdd_road_cm"); release(); return rc; }
  release();
  if (h[2] != 0 || h[3] != 0) return LBDD_ERR_ARG;   // a demand node no center reaches
  return LBDD_OK;
}
