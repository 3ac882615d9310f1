// kss_regrid.cu -- regrid steps (1)-(2) on the GPU (include/kss.h): the tagging tiles
// within `buffer` cells of a refine-flagged cell are marked, and the marked tiles are
// clustered into rectangular boxes by the signature method of Berger & Rigoutsos (the
// clustering the paper's regridding routine cites, section "Adaptive refinement and
// parallel processing"), breadth first: one cluster of CTAs walks all levels, a warp per box.
//
// Clustering rules (all integer except one efficiency comparison in FP64), for a box:
//   1. signatures sx[i] = marked tiles of column i, sy[j] = of row j;
//   2. no mark: drop; else shrink to the bounding box of the marks;
//   3. accept if marks >= efficiency * area (FP64), or if the box is a single tile;
//   4. else cut at the interior hole (zero signature) nearest the centre (ties: x before
//      y, lower index first), leaving the hole out of both halves;
//   5. else at the strongest inflection of d[i] = s[i-1] - 2 s[i] + s[i+1]: a cut between
//      i and i+1 with d[i] d[i+1] < 0, strength |d[i+1] - d[i]| (ties: cut nearest the
//      centre, then x before y, then lower index);
//   6. else bisect the longer side (x if equal) at x0 + w / 2.
// Children of a level enter the next level in order (lower half first); accepted boxes
// are appended level by level in list order, so the result is deterministic.
#include <algorithm>
#include <cstdint>
#include <cstring>
#include <new>
#include <string>

#include "runtime.h"

using namespace kss_rt;

namespace {

constexpr int kMaxSide = 8192;  // tiles per side (the codes of cluster_box have 13 bits for one)

struct alignas(16) Box {
  int x0, y0, x1, y1;
};

// ---- kernels ----

// mask[ty][tx] = 1 if a cell within `buffer` cells (periodic) of tile (tx, ty) has the
// refine flag.  A CTA takes 32 tiles of a tile row; its eight warps share out the rows
// around them, a lane reading one tile's bytes of a row (in 8-byte words where the rows are
// 8-byte aligned) and then the buffer's on both sides.  256 x 256 tiles: 86 us with one
// thread per tile, its cells one by one through two divisions each; now 13 us.
__global__ void __launch_bounds__(256) tile_mask_kernel(const uint8_t* __restrict__ flags,
                                                        long long pitch, int nx, int ny, int tile,
                                                        int buffer, int ntx, int nty, bool words,
                                                        uint8_t* __restrict__ mask) {
  __shared__ int s_any[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int tx = blockIdx.x * 32 + lane;
  for (int ty = blockIdx.y; ty < nty; ty += gridDim.y) {
    if (warp == 0) s_any[lane] = 0;
    __syncthreads();
    if (tx < ntx) {
      const int x0 = tx * tile, x1 = min(x0 + tile, nx);
      const int ya = ty * tile - buffer, yb = min((ty + 1) * tile, ny) + buffer;
      bool any = false;
      for (int y = ya + warp; y < yb && !any; y += 8) {
        int yy = y;
        if (yy < 0 || yy >= ny) yy = ((yy % ny) + ny) % ny;
        const uint8_t* const row = flags + (long long)yy * pitch;
        uint32_t bits = 0;
        if (words && x1 - x0 == tile) {
          for (int x = x0; x < x1; x += 8) {
            const uint2 w = *reinterpret_cast<const uint2*>(row + x);
            bits |= w.x | w.y;
          }
          bits &= 0x01010101u;
        } else {
          for (int x = x0; x < x1; ++x) bits |= row[x] & 1u;
        }
        for (int d = 1; d <= buffer && !bits; ++d) {
          int l = x0 - d, r = x1 - 1 + d;
          if (l < 0) l = (l % nx + nx) % nx;
          if (r >= nx) r %= nx;
          bits = (row[l] | row[r]) & 1u;
        }
        any = bits != 0;
      }
      if (any) s_any[lane] = 1;
    }
    __syncthreads();
    if (warp == 0 && tx < ntx) mask[(long long)ty * ntx + tx] = uint8_t(s_any[lane]);
  }
}

// Prefix sums of the mask along one direction: out[k][l] = marked tiles of line l at
// positions below k, k = 0 .. len.  A CTA of 32 warps takes 32 lines (a lane each); a warp
// counts 32 positions at a time, and the warps' totals are added in shared memory.
__device__ __forceinline__ void prefix_lines(const uint8_t* __restrict__ mask, int line0,
                                             int nlines, int len, long long line_stride,
                                             long long pos_stride, int* __restrict__ out) {
  __shared__ int s_tot[32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int line = line0 + lane;
  const bool ok = line < nlines;
  const uint8_t* const src = mask + line * line_stride;
  int base = 0;
  for (int p0 = 0; p0 < len; p0 += 1024) {  // (uniform over the CTA)
    const int p = p0 + 32 * warp, n = max(0, min(32, len - p));
    uint32_t bits = 0;
    if (ok) {
#pragma unroll 8
      for (int k = 0; k < n; ++k) bits |= uint32_t(src[(p + k) * pos_stride]) << k;
    }
    s_tot[warp][lane] = __popc(bits);
    __syncthreads();
    int before = base, all = 0;
    for (int w = 0; w < 32; ++w) {
      const int t = s_tot[w][lane];
      if (w < warp) before += t;
      all += t;
    }
    if (ok) {
      for (int k = 0; k < n; ++k)
        out[(long long)(p + k) * nlines + line] = before + __popc(bits & ((1u << k) - 1u));
    }
    base += all;
    __syncthreads();
  }
  if (ok && warp == 0) out[(long long)len * nlines + line] = base;
}

// pc[j][i] = marked tiles of column i in rows < j ((nty + 1) x ntx), pr[i][j] = of row j in
// columns < i ((ntx + 1) x nty): the first `column_ctas` CTAs take the columns, the others
// the rows.
__global__ void __launch_bounds__(1024) mask_prefix_kernel(const uint8_t* __restrict__ mask,
                                                           int ntx, int nty, int column_ctas,
                                                           int* __restrict__ pc,
                                                           int* __restrict__ pr) {
  const int c = blockIdx.x;
  if (c < column_ctas)
    prefix_lines(mask, 32 * c, ntx, nty, 1, ntx, pc);
  else
    prefix_lines(mask, 32 * (c - column_ctas), nty, ntx, ntx, 1, pr);
}

__device__ __forceinline__ int tile_key(int i, int lo, int hi) { return abs(2 * i - (lo + hi - 1)); }
__device__ __forceinline__ int cut_key(int i, int lo, int hi) { return abs(2 * i - (lo + hi)); }

__device__ __forceinline__ Box load_box(const Box* p) {
  const int4 v = __ldcg(reinterpret_cast<const int4*>(p));
  return Box{v.x, v.y, v.z, v.w};
}
__device__ __forceinline__ void store_box(Box* p, Box b) {
  *reinterpret_cast<int4*>(p) = make_int4(b.x0, b.y0, b.x1, b.y1);
}

// One box by one warp (rules 1 to 6 above): 0 dropped, 1 accepted (k0 the shrunk box), 2
// split into k0 and k1.  sig: room for kSig signature values; longer boxes read theirs from
// the prefix sums each time.  Every choice is the minimum of a code that orders the
// candidates by the rule's key and its ties: sides and positions are below 2^13, keys at
// most 2^14, inflection strengths at most 2^15.
constexpr int kSig = 512;
__device__ __forceinline__ int cluster_box(const int* __restrict__ pc, const int* __restrict__ pr,
                                           int ntx, int nty, Box b, double efficiency, int* sig,
                                           Box& k0, Box& k1) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int w = b.x1 - b.x0, h = b.y1 - b.y0;
  const bool fits = w + h <= kSig;
  auto value = [&](int k) {  // signature k: column x0 + k, then row y0 + k - w
    if (k < w) {
      const int* const c = pc + b.x0 + k;
      return c[(long long)b.y1 * ntx] - c[(long long)b.y0 * ntx];
    }
    const int* const r = pr + b.y0 + k - w;
    return r[(long long)b.x1 * nty] - r[(long long)b.x0 * nty];
  };
  auto at = [&](int k) { return fits ? sig[k] : value(k); };
  int ia = w, ib = -1, ja = h, jb = -1, total = 0;
  for (int k = lane; k < w + h; k += 32) {
    const int v = value(k);
    if (fits) sig[k] = v;
    if (v && k < w) {
      ia = min(ia, k);
      ib = k;
      total += v;
    } else if (v) {
      ja = min(ja, k - w);
      jb = k - w;
    }
  }
  total = __reduce_add_sync(kAll, total);
  if (total == 0) return 0;
  ia = __reduce_min_sync(kAll, ia);
  ib = __reduce_max_sync(kAll, ib);
  ja = __reduce_min_sync(kAll, ja);
  jb = __reduce_max_sync(kAll, jb);
  __syncwarp();  // the signatures are in shared memory
  const int x0 = b.x0 + ia, x1 = b.x0 + ib + 1, y0 = b.y0 + ja, y1 = b.y0 + jb + 1;
  const int n[2] = {x1 - x0, y1 - y0}, first[2] = {ia, w + ja};
  const int lo[2] = {x0, y0}, hi[2] = {x1, y1};
  if (double(total) >= efficiency * double((long long)n[0] * n[1]) || (n[0] == 1 && n[1] == 1)) {
    k0 = Box{x0, y0, x1, y1};
    return 1;
  }
  // 4. interior holes: (key, x before y, position)
  unsigned best = kAll;
#pragma unroll
  for (int a = 0; a < 2; ++a)
    for (int k = 1 + lane; k < n[a] - 1; k += 32)
      if (at(first[a] + k) == 0)
        best = min(best, unsigned(tile_key(lo[a] + k, lo[a], hi[a])) << 14 | unsigned(a) << 13 |
                             unsigned(k));
  best = __reduce_min_sync(kAll, best);
  int axis, cut, skip = 0;
  if (best != kAll) {
    axis = (best >> 13) & 1;
    cut = lo[axis] + int(best & 8191u);
    skip = 1;
  } else {
    // 5. strongest inflection: (strength down, key, x before y, position)
    unsigned c1 = kAll, c2 = kAll;
#pragma unroll
    for (int a = 0; a < 2; ++a)
      for (int k = 1 + lane; k < n[a] - 2; k += 32) {
        const int s0 = at(first[a] + k - 1), s1 = at(first[a] + k), s2 = at(first[a] + k + 1),
                  s3 = at(first[a] + k + 2);
        const int dk = s0 - 2 * s1 + s2, dk1 = s1 - 2 * s2 + s3;
        if ((dk > 0 && dk1 < 0) || (dk < 0 && dk1 > 0)) {
          const unsigned c = unsigned(32768 - abs(dk1 - dk)) << 15 |
                             unsigned(cut_key(lo[a] + k + 1, lo[a], hi[a]));
          if (c < c1) {
            c1 = c;
            c2 = unsigned(a) << 13 | unsigned(k);
          }
        }
      }
    const unsigned m = __reduce_min_sync(kAll, c1);
    c2 = __reduce_min_sync(kAll, c1 == m ? c2 : kAll);
    if (m != kAll) {
      axis = (c2 >> 13) & 1;
      cut = lo[axis] + int(c2 & 8191u) + 1;
    } else {
      // 6. bisection of the longer side
      axis = n[0] >= n[1] ? 0 : 1;
      cut = lo[axis] + n[axis] / 2;
    }
  }
  if (axis == 0) {
    k0 = Box{x0, y0, cut, y1};
    k1 = Box{cut + skip, y0, x1, y1};
  } else {
    k0 = Box{x0, y0, x1, cut};
    k1 = Box{x0, cut + skip, x1, y1};
  }
  return 2;
}

// The whole clustering, breadth first, in one cluster of CTAs: a level's boxes are shared out
// to the CTAs in contiguous runs and to their warps; after a cluster barrier every CTA knows
// how many boxes the ones before it accepted and split, and writes its own accepted boxes
// and halves in list order.  The results are those of one list processed in order.  (A
// level was two launches, whose first had one thread walk every box: 256 x 256 tiles,
// 985 boxes, 24 levels: 427 us; now 190, both by ncu.)
constexpr int kCtas = 8;
__global__ void __launch_bounds__(1024) cluster_kernel(const int* __restrict__ pc,
                                                       const int* __restrict__ pr, int ntx,
                                                       int nty, double efficiency, Box* list0,
                                                       Box* list1, Box* acc, Box* kids,
                                                       Box* result, int result_cap, int* count) {
  extern __shared__ int s_sig[];  // kSig values per warp
  __shared__ int s_tot[2];                   // accepted, split boxes of this CTA
  __shared__ int s_all[kCtas][2];            // of every CTA
  __shared__ int s_warp[32][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = int(kss::cluster_rank());
  Box* lists[2] = {list0, list1};
  int n = 1, nres = 0, cur = 0;
  // every level splits some box, and a box splits at most w + h - 2 times on any path
  for (int level = 0; n > 0 && level <= ntx + nty + 2; ++level) {
    const int per = (n + kCtas - 1) / kCtas;
    const int lo = min(rank * per, n), hi = min(lo + per, n);
    if (threadIdx.x < 2) s_tot[threadIdx.x] = 0;
    __syncthreads();
    for (int bi = lo + warp; bi < hi; bi += 32) {
      const Box b = level == 0 ? Box{0, 0, ntx, nty} : load_box(lists[cur] + bi);
      Box k0{-1, -1, -1, -1}, k1 = k0;
      const int what = cluster_box(pc, pr, ntx, nty, b, efficiency, s_sig + kSig * warp, k0, k1);
      __syncwarp();  // the signatures are rewritten by the warp's next box
      if (lane == 0) {
        const Box none{-1, -1, -1, -1};
        store_box(acc + bi, what == 1 ? k0 : none);
        store_box(kids + 2 * (long long)bi, what == 2 ? k0 : none);
        store_box(kids + 2 * (long long)bi + 1, k1);
        if (what) atomicAdd(&s_tot[what - 1], 1);
      }
    }
    __syncthreads();
    if (threadIdx.x < 2 * kCtas) {  // this CTA's totals into every CTA's table
      const uint32_t a = static_cast<uint32_t>(
          __cvta_generic_to_shared(&s_all[rank][threadIdx.x & 1]));
      uint32_t r;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                   : "=r"(r) : "r"(a), "r"(uint32_t(threadIdx.x >> 1)));
      asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(r), "r"(s_tot[threadIdx.x & 1])
                   : "memory");
    }
    __syncwarp();
    kss::cluster_arrive();
    kss::cluster_wait();
    int at_acc = nres, at_kid = 0, all_acc = 0, all_split = 0;
    for (int c = 0; c < kCtas; ++c) {
      if (c < rank) {
        at_acc += s_all[c][0];
        at_kid += 2 * s_all[c][1];
      }
      all_acc += s_all[c][0];
      all_split += s_all[c][1];
    }
    Box* const next = lists[cur ^ 1];
    for (int c0 = lo; c0 < hi; c0 += 1024) {  // (uniform over the CTA)
      const int bi = c0 + threadIdx.x;
      Box a{-1, 0, 0, 0}, k{-1, 0, 0, 0};
      if (bi < hi) {
        a = load_box(acc + bi);
        k = load_box(kids + 2 * (long long)bi);
      }
      const unsigned ba = __ballot_sync(0xffffffffu, a.x0 >= 0);
      const unsigned bk = __ballot_sync(0xffffffffu, k.x0 >= 0);
      if (lane == 0) {
        s_warp[warp][0] = __popc(ba);
        s_warp[warp][1] = __popc(bk);
      }
      __syncthreads();
      int pa = at_acc, pk = at_kid;
      for (int v = 0; v < 32; ++v) {
        if (v < warp) {
          pa += s_warp[v][0];
          pk += 2 * s_warp[v][1];
        }
        at_acc += s_warp[v][0];
        at_kid += 2 * s_warp[v][1];
      }
      const unsigned below = (1u << lane) - 1u;
      pa += __popc(ba & below);
      pk += 2 * __popc(bk & below);
      if (a.x0 >= 0 && pa < result_cap) store_box(result + pa, a);
      if (k.x0 >= 0) {
        store_box(next + pk, k);
        store_box(next + pk + 1, load_box(kids + 2 * (long long)bi + 1));
      }
      __syncthreads();
    }
    nres += all_acc;
    n = 2 * all_split;
    cur ^= 1;
    __syncwarp();
    kss::cluster_arrive();  // the next list is complete, and every CTA has read the totals
    kss::cluster_wait();
  }
  if (rank == 0 && threadIdx.x == 0) *count = nres;
}

// The tile mask, the first `room` boxes (at most `max_boxes`) and the box count to the
// caller's arrays or page-locked memory (nullptr: not wanted; a caller's boxes may be 4-byte
// aligned only).
__global__ void regrid_out_kernel(const uint8_t* __restrict__ mask, int ntiles,
                                  uint8_t* __restrict__ mask_out, const Box* __restrict__ result,
                                  const int* __restrict__ count, int room,
                                  kss_box* __restrict__ boxes_out, int* __restrict__ count_out) {
  const int t0 = blockIdx.x * blockDim.x + threadIdx.x, nt = gridDim.x * blockDim.x;
  const int n = *count;
  if (mask_out)
    for (int t = t0; t < ntiles; t += nt) mask_out[t] = mask[t];
  if (boxes_out)
    for (int t = t0; t < min(n, room); t += nt)
      boxes_out[t] = kss_box{result[t].x0, result[t].y0, result[t].x1, result[t].y1};
  if (t0 == 0 && count_out) *count_out = n;
}

// ---- host side ----

// Workspace of one tile grid, kept by a lattice between calls.
struct Workspace {
  int ntx = 0, nty = 0;
  int cap = 0;            // boxes the result holds
  Box* level[2] = {nullptr, nullptr};
  Box* acc = nullptr;     // [cap]
  Box* kids = nullptr;    // [2 cap]
  Box* result = nullptr;  // [cap]
  int* count = nullptr;
  uint8_t* mask = nullptr;
  int* pc = nullptr;      // column prefix sums [(nty + 1) ntx]
  int* pr = nullptr;      // row prefix sums [(ntx + 1) nty]
  void release() {
    void* b[] = {level[0], level[1], acc, kids, result, count, mask, pc, pr};
    for (void* p : b)
      if (p) kss_rt::dev_free(p);
    *this = Workspace{};
  }
};

cudaError_t ws_setup(Workspace& ws, int ntx, int nty) {
  if (ws.ntx == ntx && ws.nty == nty) return cudaSuccess;
  ws.release();
  const int ntiles = ntx * nty;
  ws.cap = ntiles + 1;
  const size_t bb = sizeof(Box) * size_t(ws.cap);
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.level[0], 2 * bb);
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.level[1], 2 * bb);
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.acc, bb);
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.kids, 2 * bb);
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.result, bb);
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.count, sizeof(int));
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.mask, size_t(ntiles));
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.pc, sizeof(int) * size_t(nty + 1) * ntx);
  if (e == cudaSuccess) e = kss_rt::dev_malloc(&ws.pr, sizeof(int) * size_t(nty) * (ntx + 1));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             32 * kSig * int(sizeof(int)));
  if (e != cudaSuccess) {
    cudaGetLastError();
    ws.release();
    return e;
  }
  ws.ntx = ntx;
  ws.nty = nty;
  return e;
}

// The whole regrid on device flags; outputs to host or device pointers.  L: the lattice
// whose flags these are, or nullptr.
int regrid_run(Workspace& ws, const uint8_t* d_flags, long long pitch, int nx, int ny, int tile,
               int buffer, double efficiency, uint8_t* tile_mask, kss_box* boxes,
               int32_t max_boxes, int32_t* nboxes, int on_device, cudaStream_t s, kss_lattice* L,
               std::string* msg) {
  const int ntx = (nx + tile - 1) / tile, nty = (ny + tile - 1) / tile;
  if (ntx > kMaxSide || nty > kMaxSide) return KSS_ERR_UNSUPPORTED;
  const int ntiles = ntx * nty;
  auto fail_cuda = [&](cudaError_t e) {
    if (msg) *msg = std::string("regrid: ") + cudaGetErrorString(e);
    cudaGetLastError();
    return KSS_ERR_CUDA;
  };
  cudaError_t e = ws_setup(ws, ntx, nty);
  if (e == cudaErrorMemoryAllocation) return KSS_ERR_OOM;
  if (e != cudaSuccess) return fail_cuda(e);
  const bool words = pitch % 8 == 0 && reinterpret_cast<uintptr_t>(d_flags) % 8 == 0;
  tile_mask_kernel<<<dim3((ntx + 31) / 32, nty), 256, 0, s>>>(d_flags, pitch, nx, ny, tile, buffer,
                                                             ntx, nty, words, ws.mask);
  if ((e = cudaGetLastError()) != cudaSuccess) return fail_cuda(e);
  const int cc = (ntx + 31) / 32, rc = (nty + 31) / 32;
  mask_prefix_kernel<<<cc + rc, 1024, 0, s>>>(ws.mask, ntx, nty, cc, ws.pc, ws.pr);
  if ((e = cudaGetLastError()) != cudaSuccess) return fail_cuda(e);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(kCtas);
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = 32 * kSig * sizeof(int);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCtas;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, cluster_kernel, (const int*)ws.pc, (const int*)ws.pr, ntx, nty,
                         efficiency, ws.level[0], ws.level[1], ws.acc, ws.kids, ws.result, ws.cap,
                         ws.count);
  if (e != cudaSuccess) return fail_cuda(e);
  // the outputs: this device's arrays are written directly; host ones go through borrowed
  // page-locked memory (16 bytes for the count, the mask, then boxes) where they fit; the
  // rest through the driver's copy
  static_assert(sizeof(Box) == sizeof(kss_box), "box layout");
  HostLease lease(s);
  const size_t at_boxes = 16 + (size_t(ntiles) + 15) / 16 * 16;
  unsigned char* const mail = static_cast<unsigned char*>(lease.room(at_boxes));
  int* const count_mail = static_cast<int*>(lease.room(16));
  const int wanted = std::min(max_boxes, ws.cap);
  int room = wanted;
  uint8_t* mo = nullptr;
  kss_box* bo = nullptr;
  int device = 0;
  if (on_device && (e = cudaGetDevice(&device)) != cudaSuccess) return fail_cuda(e);
  const bool direct = on_device && kernel_may_write(tile_mask, 1, device) &&
                      kernel_may_write(boxes, alignof(kss_box), device);
  if (direct) {
    mo = tile_mask;
    bo = boxes;
  } else if (mail && !on_device) {
    room = std::min<size_t>(wanted, (HostLease::kBytes - HostLease::kMailBytes - at_boxes) / sizeof(Box));
    mo = tile_mask ? mail + 16 : nullptr;
    bo = boxes ? reinterpret_cast<kss_box*>(mail + at_boxes) : nullptr;
  }
  regrid_out_kernel<<<std::max(1, std::min(64, (ntiles + 255) / 256)), 256, 0, s>>>(
      ws.mask, ntiles, mo, ws.result, ws.count, room, bo, count_mail);
  if ((e = cudaGetLastError()) != cudaSuccess) return fail_cuda(e);
  int total = 0;
  if (!count_mail &&
      (e = cudaMemcpyAsync(&total, ws.count, sizeof(int), cudaMemcpyDeviceToHost, s)) != cudaSuccess)
    return fail_cuda(e);
  if (L) {
    if (const int r = finish(L, lease)) return r;
  } else {
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return fail_cuda(e);
    lease.settled();
  }
  if (count_mail) total = *count_mail;
  if (!direct) {
    const int ncopy = std::min(total, wanted), have = bo ? std::min(ncopy, room) : 0;
    if (mo) std::memcpy(tile_mask, mail + 16, size_t(ntiles));
    if (bo) std::memcpy(boxes, mail + at_boxes, sizeof(Box) * size_t(have));
    const cudaMemcpyKind kind = on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost;
    const bool more = boxes && ncopy > have;
    if (more && (e = cudaMemcpyAsync(boxes + have, ws.result + have,
                                     sizeof(Box) * size_t(ncopy - have), kind, s)) != cudaSuccess)
      return fail_cuda(e);
    if (tile_mask && !mo &&
        (e = cudaMemcpyAsync(tile_mask, ws.mask, size_t(ntiles), kind, s)) != cudaSuccess)
      return fail_cuda(e);
    if ((more || (tile_mask && !mo)) && (e = cudaStreamSynchronize(s)) != cudaSuccess)
      return fail_cuda(e);
  }
  *nboxes = total;
  return KSS_OK;
}

bool valid_args(int tile, int buffer, double efficiency, int32_t max_boxes, int32_t* nboxes) {
  return (tile == 8 || tile == 16 || tile == 32 || tile == 64) && buffer >= 0 &&
         buffer <= 1024 && efficiency >= 0.0 && efficiency <= 1.0 && max_boxes >= 0 && nboxes;
}

}  // namespace

namespace kss_rt {
void regrid_release(kss_lattice* L) {
  if (!L || !L->regrid) return;
  Workspace* R = static_cast<Workspace*>(L->regrid);
  R->release();
  delete R;
  L->regrid = nullptr;
}
}  // namespace kss_rt

extern "C" {

int kss_regrid(kss_lattice* L, int32_t buffer, double efficiency, uint8_t* tile_mask,
               kss_box* boxes, int32_t max_boxes, int32_t* nboxes, int on_device) {
  const kss_rt::NvtxRange nvtx_range("kss_regrid");
  int rc = enter(L);
  if (rc) return rc;
  if (!valid_args(L->cfg.tile, buffer, efficiency, max_boxes, nboxes))
    return fail(L, KSS_ERR_ARG, "invalid regrid argument");
  DeviceGuard g(L->device);
  // the flags of the current step (evaluated if this step had no outputs)
  if ((rc = ensure_flags(L))) return rc;
  if (!L->regrid) {
    L->regrid = new (std::nothrow) Workspace();
    if (!L->regrid) return fail(L, KSS_ERR_OOM, "regrid workspace");
  }
  rc = regrid_run(*static_cast<Workspace*>(L->regrid), L->flags, L->pitch, L->cfg.nx, L->cfg.ny,
                  L->cfg.tile, buffer, efficiency, tile_mask, boxes, max_boxes, nboxes, on_device,
                  L->stream, L, &L->msg);
  if (rc == KSS_ERR_CUDA) L->err = rc;  // sticky
  return rc;
}

int kss_regrid_flags(const uint8_t* flags, int32_t nx, int32_t ny, int32_t tile, int32_t buffer,
                     double efficiency, uint8_t* tile_mask, kss_box* boxes, int32_t max_boxes,
                     int32_t* nboxes, int on_device, void* stream) {
  if (!flags || nx < 1 || ny < 1 || (long long)nx * ny > 0x7fffffffLL) return KSS_ERR_ARG;
  if (!valid_args(tile, buffer, efficiency, max_boxes, nboxes)) return KSS_ERR_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const uint8_t* d = flags;
  uint8_t* staged = nullptr;
  const size_t bytes = size_t(nx) * ny;
  if (!on_device) {
    if (kss_rt::dev_malloc(&staged, bytes) != cudaSuccess) {
      cudaGetLastError();
      return KSS_ERR_OOM;
    }
    if (cudaMemcpyAsync(staged, flags, bytes, cudaMemcpyHostToDevice, s) != cudaSuccess) {
      cudaGetLastError();
      kss_rt::dev_free(staged);
      return KSS_ERR_CUDA;
    }
    d = staged;
  }
  Workspace R;
  const int rc = regrid_run(R, d, nx, nx, ny, tile, buffer, efficiency, tile_mask, boxes, max_boxes,
                            nboxes, on_device, s, nullptr, nullptr);
  cudaStreamSynchronize(s);
  R.release();
  if (staged) kss_rt::dev_free(staged);
  return rc;
}

}  // extern "C"
