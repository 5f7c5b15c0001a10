// md_noalloc.cu -- md_forces_noalloc: forces of one configuration with no
// device allocation at all.
//
// Some callers cannot call cudaMalloc: code that enqueues work while a CUDA
// stream is being captured into a graph (a cudaMalloc there is illegal or
// silently leaves the graph), plugins and real-time loops that must not take
// the allocator's implicit device synchronisation, and hosts that hand the
// library a fixed memory budget they own. For them this entry point keeps all
// of its scratch (cell counts, cell starts, the cell-sorted index, per-block
// partial sums) in one file-scope device array of fixed size, allocated when
// the library is loaded and held until the process exits. The caller passes
// device pointers for every input and output.
//
// Arithmetic: all FP64, the same pair term and minimum-image rule as the FP64
// path of md_forces. One CTA per cell stages the members of the 27 cells around
// it in shared memory (every particle, when fewer than 3 cells fit per box
// edge), tests them in FP32 and evaluates in FP64 what may lie in the cutoff.
#include <cmath>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <string>

#include "kamd.h"
#include "md_device.cuh"
#include "md_internal.cuh"

namespace {

constexpr int64_t kMaxParticles = 131072;  // 2^17
constexpr int kMaxCells = 32768;
constexpr int kMaxCellsPerEdge = 32;  // kMaxCells = 32^3
constexpr int kBlock = 256;
constexpr int kMaxBlocks = 8192;  // CTAs of k_forces (their partial sums lie in `cursor`, free by then)
constexpr int kMaxTypes = 4;
constexpr int kCand = 768;        // candidates that a CTA of k_forces stages at a time
constexpr int kHits = 128;        // places of a particle's queue
constexpr int kForceThreads = 128;
constexpr int kItem = 32;         // particles of a work item at most (a warp of k_order, two turns of k_forces)
constexpr int kMaxItems = kMaxCells + (int)(kMaxParticles / kItem);

// Scratch layout (bytes): cellof[n] i32 | count[cells] i32, then the cells' first
// items | start[cells+1] i32 | cursor[cells] i32, then partial[blocks][2] f64 |
// sorted[n] i32 | items i32 | ticket u32, number of items i32
constexpr size_t kOffCellof = 0;
constexpr size_t kOffCount = kOffCellof + 4 * kMaxParticles;
constexpr size_t kOffStart = kOffCount + 4 * kMaxCells;
constexpr size_t kOffCursor = kOffStart + 4 * (kMaxCells + 1) + 12;  // keep 16-byte alignment below
constexpr size_t kOffSorted = kOffCursor + 4 * kMaxCells;
constexpr size_t kOffItems = kOffSorted + 4 * kMaxParticles;
constexpr size_t kOffTicket = (kOffItems + 4 * (size_t)kMaxItems + 255) / 256 * 256;
static_assert(kMaxCells <= 1 << 15 && kMaxParticles / kItem <= 1 << 16, "an item is one word: cell, part << 15");
static_assert(kOffCursor % 16 == 0 && 16 * (size_t)kMaxBlocks <= 4 * (size_t)kMaxCells, "partial sums fit in cursor");
constexpr size_t kScratchBytes = (kOffTicket + 256 + 255) / 256 * 256;

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

struct Table {
  // rc^2 (as given), 48 eps sigma^12, 24 eps sigma^6, 4 eps sigma^12, 4 eps sigma^6, V(rc); rc^2 widened, FP32:
  // sigma and the last in units of length_unit(), whose square and its inverse are used if it is not 1
  double rc2[kMaxTypes * kMaxTypes], c12[kMaxTypes * kMaxTypes], c6[kMaxTypes * kMaxTypes], e12[kMaxTypes * kMaxTypes],
      e6[kMaxTypes * kMaxTypes], vsh[kMaxTypes * kMaxTypes];
  float rcw2[kMaxTypes * kMaxTypes];
  int scaled;
  double unit, unit2, iunit2;
};

struct Scratch {
  int32_t* cellof;
  int32_t* count;
  int32_t* start;
  int32_t* cursor;
  int32_t* sorted;
  int32_t* items;
  double* part;
  unsigned int* ticket;
  int32_t* nitems;
};

Scratch carve(unsigned char* base) {
  Scratch s;
  s.cellof = reinterpret_cast<int32_t*>(base + kOffCellof);
  s.count = reinterpret_cast<int32_t*>(base + kOffCount);
  s.start = reinterpret_cast<int32_t*>(base + kOffStart);
  s.cursor = reinterpret_cast<int32_t*>(base + kOffCursor);
  s.sorted = reinterpret_cast<int32_t*>(base + kOffSorted);
  s.items = reinterpret_cast<int32_t*>(base + kOffItems);
  s.part = reinterpret_cast<double*>(base + kOffCursor);
  s.ticket = reinterpret_cast<unsigned int*>(base + kOffTicket);
  s.nitems = reinterpret_cast<int32_t*>(base + kOffTicket + 4);
  return s;
}

__device__ __forceinline__ double wrap01(double x, double L) {
  // already in [0, L) (the bit pattern of a negative number is above any positive one's)
  if ((unsigned long long)__double_as_longlong(x) < (unsigned long long)__double_as_longlong(L)) return x;
  x -= L * floor(x / L);
  if (x >= L) x -= L;
  if (x < 0.0) x = 0.0;
  return x;
}

__device__ __forceinline__ int cell_index(const double* pos, int64_t i, int nc, double L) {
  int c[3];
  for (int k = 0; k < 3; ++k) {
    const double x = wrap01(pos[3 * i + k], L);
    c[k] = min(max((int)(x * nc / L), 0), nc - 1);
  }
  return (c[2] * nc + c[1]) * nc + c[0];
}

__global__ void k_clear(Scratch s, int ncells) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += gridDim.x * blockDim.x) s.count[c] = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) *s.ticket = 0u;
}

__global__ void k_bin(Scratch s, const double* pos, int64_t n, int nc, double L) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = cell_index(pos, i, nc, L);
  s.cellof[i] = c;
  atomicAdd(&s.count[c], 1);
}

// One block: exclusive scans of the cell counts into start and cursor, and of
// the cells' numbers of work items into count. Each warp takes a run of cells, a
// lane one cell of every 32 (a run per thread read whole lines for one word:
// 1000 particles in 32^3 cells, the whole call 152 us, now 71).
__device__ __forceinline__ int2 scan_warp(int2 x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x.x, o), z = __shfl_up_sync(0xffffffffu, x.y, o);
    if (lane >= o) {
      x.x += y;
      x.y += z;
    }
  }
  return x;
}
__global__ void __launch_bounds__(1024) k_scan(Scratch s, int ncells) {
  __shared__ int2 warp_tot[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (ncells + 1023) / 1024 * 32;  // cells of a warp
  const int c0 = warp * per, c1 = min(c0 + per, ncells);
  int2 sum = make_int2(0, 0);
#pragma unroll 8
  for (int c = c0 + lane; c < c1; c += 32) {
    const int m = s.count[c];
    sum.x += m;
    sum.y += (m + kItem - 1) / kItem;
  }
  sum = make_int2(__reduce_add_sync(0xffffffffu, sum.x), __reduce_add_sync(0xffffffffu, sum.y));
  if (lane == 0) warp_tot[warp] = sum;
  __syncthreads();
  if (warp == 0) warp_tot[lane] = scan_warp(warp_tot[lane]);
  __syncthreads();
  int2 run = warp > 0 ? warp_tot[warp - 1] : make_int2(0, 0);
#pragma unroll 4
  for (int r = c0; r < c1; r += 32) {
    const int c = r + lane;
    const int m = c < c1 ? s.count[c] : 0;
    const int2 own = make_int2(m, (m + kItem - 1) / kItem), x = scan_warp(own);
    if (c < c1) {
      s.start[c] = run.x + x.x - own.x;
      s.cursor[c] = run.x + x.x - own.x;
      s.count[c] = run.y + x.y - own.y;
    }
    run.x += __shfl_sync(0xffffffffu, x.x, 31);
    run.y += __shfl_sync(0xffffffffu, x.y, 31);
  }
  if (threadIdx.x == 0) {
    s.start[ncells] = warp_tot[31].x;
    *s.nitems = warp_tot[31].y;
  }
}

// Members of each cell, in any order, and the work items: whoever takes the
// first place of a part writes it down.
__global__ void k_scatter(Scratch s, int64_t n) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int c = s.cellof[i];
  const int slot = atomicAdd(&s.cursor[c], 1);
  s.sorted[slot] = (int32_t)i;
  const int k = slot - s.start[c];
  if (k % kItem == 0) s.items[s.count[c] + k / kItem] = c | (k / kItem) << 15;
}

// One warp per work item: order the cell's members by particle index (deterministic).
__global__ void k_order(Scratch s) {
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5, items = *s.nitems;
  for (int q = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; q < items; q += warps) {
    const int c = s.items[q] & 0x7fff, e = kItem * (s.items[q] >> 15) + lane;
    const int lo = s.start[c], m = s.start[c + 1] - lo;
    const int mine = e < m ? s.sorted[lo + e] : 0x7fffffff;
    int rank = 0;
    for (int m0 = 0; m0 < m; m0 += 32) {
      const int other = m0 + lane < m ? s.sorted[lo + m0 + lane] : 0x7fffffff;
      const int lim = min(32, m - m0);
      for (int t = 0; t < lim; ++t) rank += (__shfl_sync(0xffffffffu, other, t) < mine);
    }
    // write into cellof (free after scatter) to avoid overwriting unread members
    if (e < m) s.cellof[lo + rank] = mine;
  }
}

// Forces, and the block's share of energy and virial. A work item is up to 32
// particles of one cell, or, without cells (nc == 0), 32 particles in input
// order with every particle a candidate. What bounds it is the FP64 unit (two
// operations per SM and clock): each particle has 8 lanes, which test the
// staged candidates in FP32 on 32-bit words, queue those that may lie in the
// cutoff (by ballots, in candidate order) and deal them out evenly for the FP64
// terms. Members of the 27 cells are read from memory once per cell instead of
// once per particle and pair, and wrapped once. A candidate of an unknown type
// makes every particle of the item NaN. Measured at n = 20 011 (the whole call):
// 3093 us with one thread per particle walking the cells in FP64, 190 us so.
__global__ void __launch_bounds__(kForceThreads) k_forces(Scratch s, const double* __restrict__ pos,
                                                          const uint8_t* __restrict__ types, int n, int ntypes, int nc,
                                                          double L, Table tab, double* f, double* pe_out,
                                                          double* vir_out) {
  __shared__ double cand[3][kCand];
  __shared__ uint4 word[kCand];  // x, y, z, type << 30 | index
  __shared__ uint16_t hits[kForceThreads / 8][kHits];
  __shared__ int lo_[27], base_[28];
  __shared__ Table tb;
  __shared__ double red[kForceThreads / 32][2];
  __shared__ int bad_;
  __shared__ bool last;
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 3, sl = tid & 7;
  const unsigned group = 0xffu << (lane & 24), before = group & ((1u << lane) - 1u);
  for (int t = tid; t < (int)(sizeof(Table) / 4); t += kForceThreads)
    reinterpret_cast<int*>(&tb)[t] = reinterpret_cast<const int*>(&tab)[t];
  const double to_word = 4294967296.0 / L;
  const float sc = (float)(L / 4294967296.0 / tab.unit);
  const long long hLb = __double_as_longlong(0.5 * L);
  double pe = 0.0, vir = 0.0;
  const int items = nc > 0 ? *s.nitems : (n + kItem - 1) / kItem;
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    __syncthreads();  // the previous item's shared data are read
    // runs of candidates in `cellof` (the cell order), and this item's particles
    int p0 = 0, p1 = 0;
    if (nc > 0) {
      const int cell = s.items[item] & 0x7fff;
      if (tid < 27) {
        const int cx = cell % nc, cy = (cell / nc) % nc, cz = cell / (nc * nc);
        const int c = (((cz + tid / 9 - 1 + nc) % nc) * nc + (cy + (tid / 3) % 3 - 1 + nc) % nc) * nc + (cx + tid % 3 - 1 + nc) % nc;
        lo_[tid] = s.start[c];
        base_[tid + 1] = s.start[c + 1] - s.start[c];
      }
      p0 = s.start[cell] + kItem * (s.items[item] >> 15);
      p1 = min(p0 + kItem, s.start[cell + 1]);
    } else {
      if (tid == 0) {
        lo_[0] = 0;
        base_[1] = n;
      } else if (tid < 27) {
        lo_[tid] = 0;
        base_[tid + 1] = 0;
      }
      p0 = kItem * item;
      p1 = min(p0 + kItem, n);
    }
    if (tid == 0) {
      base_[0] = 0;
      bad_ = 0;
    }
    __syncthreads();
    if (tid == 0)
      for (int k = 0; k < 27; ++k) base_[k + 1] += base_[k];
    __syncthreads();
    const int total = base_[27];
    for (int c0 = 0; c0 < total; c0 += kCand) {
      const int nst = min(kCand, total - c0);
      if (c0 > 0) __syncthreads();  // the previous candidates are read
      for (int t = tid; t < nst; t += kForceThreads) {
        int a = 0, b = 27;
        while (b - a > 1) {  // base_[a] <= c0 + t < base_[b]
          const int m = (a + b) >> 1;
          if (base_[m] <= c0 + t) a = m; else b = m;
        }
        const int q = lo_[a] + (c0 + t - base_[a]);
        const int j = nc > 0 ? s.cellof[q] : q;
        const double x = wrap01(pos[3 * (int64_t)j], L), y = wrap01(pos[3 * (int64_t)j + 1], L),
                     z = wrap01(pos[3 * (int64_t)j + 2], L);
        const unsigned tj = types[j];
        if ((int)tj >= ntypes) bad_ = 1;
        uint4 w = kamd::words_of(to_word, x, y, z, 0u);
        w.w = ((tj & 3u) << 30) | (unsigned)j;
        cand[0][t] = x;
        cand[1][t] = y;
        cand[2][t] = z;
        word[t] = w;
      }
      __syncthreads();
      // 8 lanes per particle, 16 particles at a time
      for (int q0 = p0; q0 < p1; q0 += kForceThreads / 8) {
        const bool act = q0 + g < p1;
        const int q = act ? q0 + g : p0;
        const int i = nc > 0 ? s.cellof[q] : q;
        const double xi = wrap01(pos[3 * (int64_t)i], L), yi = wrap01(pos[3 * (int64_t)i + 1], L),
                     zi = wrap01(pos[3 * (int64_t)i + 2], L);
        const uint4 wi = kamd::words_of(to_word, xi, yi, zi, 0u);
        const unsigned ty = types[i];
        const int row = ((int)ty < ntypes ? (int)ty : 0) * ntypes;
        double fx = 0.0, fy = 0.0, fz = 0.0;
        int held = 0;
        for (int t0 = 0; t0 < nst; t0 += 8) {
          bool hit = false;
          const int t = t0 + sl;
          if (act && t < nst) {
            const uint4 w = word[t];
            const float dx = (float)(int)(wi.x - w.x) * sc, dy = (float)(int)(wi.y - w.y) * sc, dz = (float)(int)(wi.z - w.z) * sc;
            const int tj = (int)(w.w >> 30);
            hit = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) < tb.rcw2[row + min(tj, ntypes - 1)] &&
                  (int)(w.w & 0x3fffffffu) != i;
          }
          const unsigned m = __ballot_sync(0xffffffffu, hit);
          if (hit) hits[g][held + __popc(m & before)] = (uint16_t)t;
          held += __popc(m & group);
          if (t0 + 8 < nst && !__any_sync(0xffffffffu, held > kHits - 8)) continue;
          __syncwarp();
          for (int k = sl; k < held; k += 8) {
            const int h = hits[g][k];
            const double dx = kamd::image_f64(xi - cand[0][h], L, hLb), dy = kamd::image_f64(yi - cand[1][h], L, hLb),
                         dz = kamd::image_f64(zi - cand[2][h], L, hLb);
            const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
            const int tt = row + min((int)(word[h].w >> 30), ntypes - 1);
            if (kamd::less_f64(r2, tb.rc2[tt])) {
              double y = kamd::rcp_f64(r2);
              if (__builtin_expect(tab.scaled, 0)) y *= tab.unit2;
              const double y3 = y * y * y;
              const double w = y3 * fma(tb.c12[tt], y3, -tb.c6[tt]);
              double fr = w * y;
              if (__builtin_expect(tab.scaled, 0)) fr *= tab.iunit2;
              fx = fma(fr, dx, fx);
              fy = fma(fr, dy, fy);
              fz = fma(fr, dz, fz);
              pe += fma(y3, fma(tb.e12[tt], y3, -tb.e6[tt]), -tb.vsh[tt]);
              vir += w;
            }
          }
          __syncwarp();
          held = 0;
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) {
          fx += __shfl_xor_sync(0xffffffffu, fx, o);
          fy += __shfl_xor_sync(0xffffffffu, fy, o);
          fz += __shfl_xor_sync(0xffffffffu, fz, o);
        }
        if (act && sl < 3) {  // (more than kCand candidates: the sums of the earlier ones are there)
          double v = sl == 0 ? fx : (sl == 1 ? fy : fz);
          double* out = f + 3 * (int64_t)i + sl;
          if (c0 > 0) v += *out;
          *out = c0 + nst >= total && bad_ ? __longlong_as_double(0x7ff8000000000000ll) : v;
        }
      }
    }
    if (bad_) pe = vir = __longlong_as_double(0x7ff8000000000000ll);
  }
  // fixed-order block sums of the half pair energies and virials
  pe = kamd::warp_sum(0.5 * pe);
  vir = kamd::warp_sum(0.5 * vir);
  if (lane == 0) {
    red[tid >> 5][0] = pe;
    red[tid >> 5][1] = vir;
  }
  __syncthreads();
  if (tid == 0) {
    double a = red[0][0], b = red[0][1];
    for (int w = 1; w < kForceThreads / 32; ++w) {
      a += red[w][0];
      b += red[w][1];
    }
    s.part[2 * blockIdx.x] = a;
    s.part[2 * blockIdx.x + 1] = b;
    __threadfence();
    last = atomicAdd(s.ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  // the last block: every block's sums, strided over the threads, then as above
  __threadfence();
  double a = 0.0, b = 0.0;
  for (unsigned k = tid; k < gridDim.x; k += kForceThreads) {
    a += __ldcg(s.part + 2 * k);
    b += __ldcg(s.part + 2 * k + 1);
  }
  a = kamd::warp_sum(a);
  b = kamd::warp_sum(b);
  if (lane == 0) {
    red[tid >> 5][0] = a;
    red[tid >> 5][1] = b;
  }
  __syncthreads();
  if (tid == 0) {
    a = red[0][0];
    b = red[0][1];
    for (int w = 1; w < kForceThreads / 32; ++w) {
      a += red[w][0];
      b += red[w][1];
    }
    if (pe_out) *pe_out = a;
    if (vir_out) *vir_out = b;
  }
}

md_status noalloc_fail(md_status st, const std::string& m) {
  kamd_set_global_error(m);
  return st;
}

// Device address of the static scratch array, per CUDA context. The host-side
// name g_noalloc_scratch is a stand-in, not a device address, and the array
// moves whenever the module is loaded again (a new context after
// cudaDeviceReset, or another context on the same device). So the address is
// looked up afresh on every call made outside a stream capture, and the
// cached value of the current context is used only while a capture is open
// (where the look-up itself is not allowed).
typedef int (*CtxGetCurrentFn)(void**);

struct ScratchSlot {
  void* ctx;
  unsigned char* ptr;
};
constexpr int kSlots = 64;
ScratchSlot g_slots[kSlots];
int g_nslots = 0;
std::mutex g_slots_mu;

CtxGetCurrentFn ctx_get_current() {
  static CtxGetCurrentFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<CtxGetCurrentFn>(f);
  }();
  return fn;
}

md_status scratch_address(cudaStream_t st, unsigned char** out) {
  CtxGetCurrentFn get = ctx_get_current();
  if (!get) return noalloc_fail(MD_ERR_CUDA, "md_forces_noalloc: cuCtxGetCurrent is not available");
  // the capture query also sets up the runtime's context on this thread if
  // nothing else has yet
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  cudaError_t e = cudaStreamIsCapturing(st, &cap);
  if (e != cudaSuccess) return noalloc_fail(MD_ERR_CUDA, std::string("cudaStreamIsCapturing: ") + cudaGetErrorString(e));
  void* ctx = nullptr;
  if (get(&ctx) != 0 || !ctx) return noalloc_fail(MD_ERR_CUDA, "md_forces_noalloc: no current CUDA context");
  std::lock_guard<std::mutex> lock(g_slots_mu);
  int k = 0;
  while (k < g_nslots && g_slots[k].ctx != ctx) ++k;
  if (cap != cudaStreamCaptureStatusNone) {
    if (k == g_nslots)
      return noalloc_fail(MD_ERR_INVALID_ARG,
                          "md_forces_noalloc: make one call in this CUDA context before capturing a stream");
    *out = g_slots[k].ptr;
    return MD_OK;
  }
  void* ptr = nullptr;
  e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
  if (e != cudaSuccess || !ptr)
    return noalloc_fail(MD_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
  if (k == g_nslots) {
    if (g_nslots == kSlots) k = 0;  // many contexts: reuse the oldest slot
    else ++g_nslots;
  }
  g_slots[k] = ScratchSlot{ctx, static_cast<unsigned char*>(ptr)};
  *out = g_slots[k].ptr;
  return MD_OK;
}

}  // namespace

extern "C" md_status md_forces_noalloc(int64_t n, const double* pos, const uint8_t* types, int ntypes, double L,
                                       const double* eps, const double* sigma, const double* rc, double* f, double* pe,
                                       double* virial, void* stream) {
  if (n < 2 || n > kMaxParticles)
    return noalloc_fail(MD_ERR_INVALID_ARG, "md_forces_noalloc: n must be in [2, 131072] (fixed scratch size)");
  if (!pos || !types || !f || !eps || !sigma || !rc)
    return noalloc_fail(MD_ERR_INVALID_ARG, "md_forces_noalloc: pos, types, f and the tables are required");
  if (ntypes < 1 || ntypes > kMaxTypes) return noalloc_fail(MD_ERR_INVALID_ARG, "md_forces_noalloc: ntypes in [1, 4]");
  if (!(L > 0) || !std::isfinite(L)) return noalloc_fail(MD_ERR_INVALID_ARG, "md_forces_noalloc: L must be > 0");
  Table tab;
  double rcmax = 0;
  for (int a = 0; a < ntypes; ++a)
    for (int b = 0; b < ntypes; ++b) {
      const int t = a * ntypes + b, u = b * ntypes + a;
      if (!(eps[t] > 0) || !(sigma[t] > 0) || !(rc[t] > 0) || eps[t] != eps[u] || sigma[t] != sigma[u] ||
          rc[t] != rc[u])
        return noalloc_fail(MD_ERR_INVALID_ARG, "md_forces_noalloc: tables must be positive and symmetric");
      if (!(rc[t] < 0.5 * L)) return noalloc_fail(MD_ERR_INVALID_ARG, "md_forces_noalloc: every cutoff must be < L/2");
      const double sr6 = std::pow(sigma[t] / rc[t], 6.0);
      tab.rc2[t] = rc[t] * rc[t];
      tab.vsh[t] = 4.0 * eps[t] * (sr6 * sr6 - sr6);
      rcmax = std::max(rcmax, rc[t]);
    }
  // the FP32 pre-test: r^2 from 32-bit words is off by less than 4 r sqrt(3) L/2^31 and a relative 1e-6
  const double u = tab.unit = length_unit(rcmax), off = std::ldexp(L, -31) / u;
  tab.scaled = u != 1.0;
  tab.unit2 = u * u;
  tab.iunit2 = 1.0 / tab.unit2;
  for (int t = 0; t < ntypes * ntypes; ++t) {
    const double s1 = sigma[t] / u, s3 = s1 * s1 * s1, s6 = s3 * s3, r = rc[t] / u;
    tab.c12[t] = 48.0 * eps[t] * s6 * s6;
    tab.c6[t] = 24.0 * eps[t] * s6;
    tab.e12[t] = 4.0 * eps[t] * s6 * s6;
    tab.e6[t] = 4.0 * eps[t] * s6;
    tab.rcw2[t] = (float)(r * r * (1.0 + 1e-5) + 4.0 * std::sqrt(3.0) * (r + off) * off);
  }
  // cells of edge >= the largest cutoff, at most kMaxCellsPerEdge per edge
  // (clamped in double, so any finite L is safe); fewer than 3: all pairs
  int nc = (int)std::min(std::floor(L / rcmax), (double)kMaxCellsPerEdge);
  if (nc < 3) nc = 1;
  const int ncells = nc * nc * nc;
  cudaStream_t st = (cudaStream_t)stream;
  unsigned char* base = nullptr;
  const md_status as = scratch_address(st, &base);
  if (as != MD_OK) return as;
  const Scratch s = carve(base);
  cudaError_t e;
  const int nb = (int)((n + kBlock - 1) / kBlock);
  // at most this many work items (their number is known on the device only)
  const int items = (int)((n + kItem - 1) / kItem) + (nc >= 3 ? (int)std::min<int64_t>(ncells, n) : 0);
  k_clear<<<std::max(1, std::min(64, (ncells + kBlock - 1) / kBlock)), kBlock, 0, st>>>(s, ncells);
  if (nc >= 3) {  // (otherwise every particle meets every other: no cells)
    k_bin<<<nb, kBlock, 0, st>>>(s, pos, n, nc, L);
    k_scan<<<1, 1024, 0, st>>>(s, ncells);
    k_scatter<<<nb, kBlock, 0, st>>>(s, n);
    k_order<<<std::min(1024, (items * 32 + kBlock - 1) / kBlock), kBlock, 0, st>>>(s);
  }
  k_forces<<<std::min(items, kMaxBlocks), kForceThreads, 0, st>>>(s, pos, types, (int)n, ntypes, nc >= 3 ? nc : 0, L, tab, f,
                                                                  pe, virial);
  e = cudaGetLastError();
  if (e != cudaSuccess) return noalloc_fail(MD_ERR_CUDA, std::string("kernel launch: ") + cudaGetErrorString(e));
  return MD_OK;
}
