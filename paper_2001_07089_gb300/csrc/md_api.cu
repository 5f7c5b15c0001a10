// md_api.cu -- the C ABI declared in include/kamd.h: system set-up, device
// memory, state transfer, and the launches of the persistent step kernel.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <unordered_map>
#include <vector>

#include "kamd.h"
#include "md_device.cuh"
#include "md_internal.cuh"

// A shape of the persistent launch, and the launch as an instantiated CUDA graph
// (one cooperative kernel node whose parameters are updated per call).
struct LaunchShape {
  int grid = 0, carveout = 0;  // CTAs; percent of the SM's shared memory that they take
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  cudaGraphNode_t gnode = nullptr;
  int g_grid = 0, g_block = 0, g_carveout = 0;
  size_t g_smem = 0;
};

struct md_system {
  // configuration
  int nrep = 0, ntypes = 0;
  int ndim = 3;         // 2: particles in the plane z = L/2, v_z = 0 (two-dimensional model)
  int64_t n_total = 0;  // particles, caller order
  int64_t ntot = 0;     // slots (padded)
  int ntiles = 0;
  bool mixed = true;
  std::vector<int64_t> n_per, out0;
  std::vector<double> L_per;
  std::vector<int64_t> n_type0;  // particles of type 0 per replica
  double eps[16] = {0}, sig[16] = {0}, rc[16] = {0};
  double mass = 1.0;
  double unit = 1.0;  // FP64 path: unit of length of its FP32 numbers (length_unit)
  md_tuning tun{4, 256, 0.3, 0.7};
  cudaStream_t stream = nullptr;
  int device = 0, nsm = 0;
  int maxrows = 0;
  int stage_cap = 0;  // candidates the list build stages per group (dynamic shared memory)
  int64_t ncells = 0;
  bool have_state = false;
  // host mirrors of the control block and the replicas (see upload_state)
  std::vector<RepDev> reps;
  CtlDev ctl{};
  bool ctl_now = true, reps_now = true;  // the mirror is as new as the device's copy, or newer
  bool reps_dirty = false;               // replicas newer here than on the device
  unsigned char* h_land = nullptr;       // pinned: where copies from the device arrive
  std::vector<unsigned char> up;         // where copies to the device are put together
  // device memory
  unsigned char* d_state = nullptr;  // the control block, then the replicas
  RepDev* d_reps = nullptr;          // (in d_state)
  int32_t* d_tile_rep = nullptr;
  CtlDev* d_ctl = nullptr;  // (in d_state)
  uint64_t* d_pfx = nullptr;
  uint4* d_pq[2] = {nullptr, nullptr};
  float* d_velf = nullptr;
  float* d_frcf = nullptr;
  uint4* d_xbq = nullptr;
  uint4* d_xbq_in = nullptr;
  double4_32a* d_p4[2] = {nullptr, nullptr};
  double* d_veld = nullptr;
  double* d_frcd = nullptr;
  int32_t* d_gid = nullptr;
  uint8_t* d_typ = nullptr;
  int32_t* d_img = nullptr;
  uint64_t* d_tpfx = nullptr;
  double4_32a* d_tp4 = nullptr;
  void* d_tvel = nullptr;
  void* d_tfrc = nullptr;
  int32_t* d_tgid = nullptr;
  uint8_t* d_ttyp = nullptr;
  int32_t* d_timg = nullptr;
  int32_t* d_cellof = nullptr;
  int32_t* d_cell_rep = nullptr;
  int32_t* d_ccount = nullptr;
  int32_t* d_cstart = nullptr;
  int32_t* d_ccursor = nullptr;
  int32_t* d_chunk = nullptr;
  int32_t* d_cta_sm = nullptr;  // SM id per CTA of the persistent grid
  int2* d_redmap = nullptr;     // reduction chunks (replica, chunk index)
  int2* d_redrep = nullptr;     // per replica (first chunk, chunks)
  double* d_redpart = nullptr;  // chunk sums
  int64_t nred = 0;
  int red2 = 0;
  int red_tiles = MD_RED_TILES;
  int cta_sm_cap = 0;
  int32_t* d_scat = nullptr;
  int32_t* d_nbr = nullptr;
  int32_t* d_nbr_in = nullptr;
  int32_t* d_nnb_in = nullptr;
  int32_t* d_nnb = nullptr;
  double* d_part[2] = {nullptr, nullptr};
  uint8_t* d_typ_caller = nullptr;
  int32_t* d_rep_of_caller = nullptr;
  double* d_msd_ref[MD_MSD_SLOTS] = {};  // unwrapped reference positions r(t_w), caller order; [0] always held
  bool msd_valid[MD_MSD_SLOTS] = {};
  ThermoDev* d_thermo = nullptr;
  int64_t thermo_cap = 0;
  double* d_io = nullptr;  // caller-order staging (n_total*3 doubles)
  int32_t* d_io_i = nullptr;
  unsigned long long* d_rdf = nullptr;
  int64_t rdf_nbins = 0;
  double rdf_dr = 0.0;
  int64_t rdf_meas = 0;
  std::vector<int32_t> rdf_blk;  // first CTA of each replica (see md_rdf)
  double* d_msd_part = nullptr;
  unsigned long long* d_count = nullptr;
  size_t bytes = 0;  // device bytes currently held (dalloc/dfree)
  std::unordered_map<const void*, size_t> alloc_sizes;
  size_t list_bytes = 0;
  unsigned long long timeout_ns = 10ull * 1000 * 1000 * 1000;
  LaunchShape shape[2];  // the usual one, and the one of as many CTAs as fit (configure_grid, wide_launch)
  bool use_graph = true;
  // partial records of NVE log steps reduced after the launch (size in doubles)
  double* d_plog = nullptr;
  longlong2* d_plog_rec = nullptr;
  size_t plog_cap = 0;
  int plog_slots = 0;
  bool log_now = false;  // KAMD_LOG_NOW=1: every log record reduced at its step
  int64_t graph_launches = 0;
  int64_t kernel_launches = 0;  // persistent launches and log-record launches
  std::string err;
};

namespace {

thread_local std::string g_create_err;

md_status fail(md_system* s, md_status code, const std::string& msg) {
  if (s) s->err = msg;
  else g_create_err = msg;
  return code;
}

md_status cuda_fail(md_system* s, cudaError_t e, const char* what) {
  std::string m = std::string(what) + ": " + cudaGetErrorString(e);
  return fail(s, e == cudaErrorMemoryAllocation ? MD_ERR_OOM : MD_ERR_CUDA, m);
}

#define CK(call)                                         \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return cuda_fail(s, e_, #call); \
  } while (0)

template <typename T>
md_status dalloc(md_system* s, T** p, size_t count) {
  *p = nullptr;
  if (count == 0) count = 1;
  cudaError_t e = cudaMalloc((void**)p, count * sizeof(T));
  if (e != cudaSuccess) return cuda_fail(s, e, "cudaMalloc");
  s->bytes += count * sizeof(T);
  s->alloc_sizes[(const void*)*p] = count * sizeof(T);
  e = cudaMemsetAsync(*p, 0, count * sizeof(T), s->stream);
  if (e != cudaSuccess) return cuda_fail(s, e, "cudaMemsetAsync");
  return MD_OK;
}

// Free a device array allocated by dalloc and take its size off the
// footprint counter (md_get_info's device_bytes).
template <typename T>
void dfree(md_system* s, T*& p) {
  if (p) {
    auto it = s->alloc_sizes.find((const void*)p);
    if (it != s->alloc_sizes.end()) {
      s->bytes -= it->second;
      s->alloc_sizes.erase(it);
    }
    cudaFree((void*)p);
  }
  p = nullptr;
}

#define CKS(call)                 \
  do {                            \
    md_status st_ = (call);       \
    if (st_ != MD_OK) return st_; \
  } while (0)

// ------------------------------------------------------------------ kernels

// Map caller-order particle g to its slot: identity order inside a replica.
__global__ void k_set_state(bool mixed, int ndim, int64_t n_total, int64_t ntot, const RepDev* reps,
                            const int32_t* rep_of, const uint8_t* typ_caller, const double* pos, const double* vel,
                            int cur, uint64_t* pfx, uint4* pq, float* velf, float* frcf, uint4* xbq, double4_32a* p4,
                            double* veld, double* frcd, int32_t* gid, uint8_t* typ, int32_t* img) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_total) return;
  const RepDev& R = reps[rep_of[g]];
  const int64_t i = R.off + (g - R.out0);
  const uint32_t t = typ_caller[g];
  double x[3];
  for (int c = 0; c < 3; ++c) x[c] = kamd::wrap_box(pos[3 * g + c], R.L);
  if (ndim == 2) x[2] = 0.5 * R.L;  // two dimensions: the plane z = L/2
  if (mixed) {
    uint32_t hi[3];
    for (int c = 0; c < 3; ++c) {
      const uint64_t u = kamd::to_fixed(x[c], R.invL);
      pfx[c * ntot + i] = u;
      hi[c] = (uint32_t)(u >> 32);
      velf[c * ntot + i] = (vel && (ndim == 3 || c < 2)) ? (float)vel[3 * g + c] : 0.0f;
      frcf[c * ntot + i] = 0.0f;
    }
    pq[i] = make_uint4(hi[0], hi[1], hi[2], t);
  } else {
    p4[i] = make_double4_32a(x[0], x[1], x[2], __longlong_as_double((long long)t));
    pq[i] = kamd::words_of(R.fx32, x[0], x[1], x[2], t);
    for (int c = 0; c < 3; ++c) {
      veld[c * ntot + i] = (vel && (ndim == 3 || c < 2)) ? vel[3 * g + c] : 0.0;
      frcd[c * ntot + i] = 0.0;
    }
  }
  xbq[i] = pq[i];
  for (int c = 0; c < 3; ++c) img[c * ntot + i] = 0;
  gid[i] = (int32_t)g;
  typ[i] = (uint8_t)t;
}

// Simple-cubic lattice with jitter (Sec. "Initialization of positions"); in
// two dimensions a square lattice in the plane z = L/2.
__global__ void k_lattice(int ndim, int64_t n_total, const RepDev* reps, const int32_t* rep_of, double jitter,
                          uint64_t seed, double* pos) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_total) return;
  const RepDev& R = reps[rep_of[g]];
  const int64_t p = g - R.out0, n = R.n;
  int64_t m = 1;
  if (ndim == 3) while (m * m * m < n) ++m;
  else while (m * m < n) ++m;
  const double a = R.L / (double)m;
  const int64_t sites = ndim == 3 ? m * m * m : m * m;
  const int64_t site = (int64_t)(((unsigned __int128)p * (unsigned __int128)sites) / (unsigned __int128)n);
  const int64_t k[3] = {site % m, (site / m) % m, site / (m * m)};
  double u[3];
  kamd::jitter3(seed, (uint32_t)p, u);
  for (int c = 0; c < 3; ++c) {
    double x = (ndim == 2 && c == 2) ? 0.5 * R.L : (0.5 + (double)k[c]) * a + jitter * u[c];
    if (x >= R.L) x -= R.L;
    else if (x < 0.0) x += R.L;
    pos[3 * g + c] = x;
  }
}

__global__ void k_get_state(bool mixed, int64_t ntot, const RepDev* reps, const int32_t* tile_rep, int cur,
                            const uint64_t* pfx, const float* velf, const double4_32a* p4, const double* veld,
                            const int32_t* gid, const int32_t* img, double* pos, double* vel, int32_t* imgo) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntot) return;
  const RepDev& R = reps[tile_rep[i >> 5]];
  if (i - R.off >= R.n) return;
  const int64_t g = gid[i];
  for (int c = 0; c < 3; ++c) {
    if (pos) pos[3 * g + c] = mixed ? kamd::from_fixed(pfx[c * ntot + i], R.L) : (c == 0 ? p4[i].x : c == 1 ? p4[i].y : p4[i].z);
    if (vel) vel[3 * g + c] = mixed ? (double)velf[c * ntot + i] : veld[c * ntot + i];
    if (imgo) imgo[3 * g + c] = img[c * ntot + i];
  }
}

__global__ void k_get_forces(bool mixed, int64_t ntot, const RepDev* reps, const int32_t* tile_rep, const float* frcf,
                             const double* frcd, const int32_t* gid, double* f) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntot) return;
  const RepDev& R = reps[tile_rep[i >> 5]];
  if (i - R.off >= R.n) return;
  const int64_t g = gid[i];
  for (int c = 0; c < 3; ++c) f[3 * g + c] = mixed ? (double)frcf[c * ntot + i] : frcd[c * ntot + i];
}

__global__ void k_set_images(int64_t n_total, int64_t ntot, const RepDev* reps, const int32_t* rep_of,
                             const int32_t* imgs, int32_t* img) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_total) return;
  const RepDev& R = reps[rep_of[g]];
  const int64_t i = R.off + (g - R.out0);
  for (int c = 0; c < 3; ++c) img[c * ntot + i] = imgs[3 * g + c];
}

// Unwrapped caller-order positions x + L*image (MSD reference / current).
__global__ void k_unwrapped(bool mixed, int64_t ntot, const RepDev* reps, const int32_t* tile_rep, const uint64_t* pfx,
                            const double4_32a* p4, const int32_t* gid, const int32_t* img, double* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntot) return;
  const RepDev& R = reps[tile_rep[i >> 5]];
  if (i - R.off >= R.n) return;
  const int64_t g = gid[i];
  for (int c = 0; c < 3; ++c) {
    const double x = mixed ? kamd::from_fixed(pfx[c * ntot + i], R.L) : (c == 0 ? p4[i].x : c == 1 ? p4[i].y : p4[i].z);
    out[3 * g + c] = x + R.L * (double)img[c * ntot + i];
  }
}

// Sums of squared displacement per type (Eq. (msdwithi)), one record of sums
// and counts per CTA: each thread adds up its particles, then warp trees and the
// CTA's warps in order. The grid is fixed by the number of tiles, so the order
// of every sum is too. (One record per tile, added up by a single thread, took
// 3.5 ms at N = 10^6.)
#define MSD_THREADS 256
#define MSD_BLOCKS 1024
__device__ __forceinline__ void msd_reduce(const double* v, const double* cnt, int ntypes, double* out) {
  __shared__ double red[MSD_THREADS / 32][2 * MD_MAXTYPES];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int a = 0; a < ntypes; ++a) {
    const double x = kamd::warp_sum(v[a]), y = kamd::warp_sum(cnt[a]);
    if (lane == 0) {
      red[warp][a] = x;
      red[warp][MD_MAXTYPES + a] = y;
    }
  }
  __syncthreads();
  if (threadIdx.x < 2 * MD_MAXTYPES && (threadIdx.x & (MD_MAXTYPES - 1)) < ntypes) {
    double t = red[0][threadIdx.x];
    for (int w = 1; w < MSD_THREADS / 32; ++w) t += red[w][threadIdx.x];
    out[threadIdx.x] = t;
  }
}
__global__ void __launch_bounds__(MSD_THREADS) k_msd_blocks(bool mixed, int ntypes, int64_t ntot, const RepDev* reps,
                                                            const int32_t* tile_rep, const uint64_t* pfx,
                                                            const double4_32a* p4, const int32_t* gid, const uint8_t* typ,
                                                            const int32_t* img, const double* ref, double* part) {
  double v[MD_MAXTYPES] = {0, 0, 0, 0};
  double cnt[MD_MAXTYPES] = {0, 0, 0, 0};
  int n[MD_MAXTYPES] = {0, 0, 0, 0};
  for (int64_t i = (int64_t)blockIdx.x * MSD_THREADS + threadIdx.x; i < ntot; i += (int64_t)gridDim.x * MSD_THREADS) {
    const RepDev& R = reps[tile_rep[i >> 5]];
    if (i - R.off >= R.n) continue;
    const int64_t g = gid[i];
    const int t = typ[i];
    double d2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      const double x = mixed ? kamd::from_fixed(pfx[c * ntot + i], R.L) : (c == 0 ? p4[i].x : c == 1 ? p4[i].y : p4[i].z);
      const double d = x + R.L * (double)img[c * ntot + i] - ref[3 * g + c];
      d2 += d * d;
    }
#pragma unroll
    for (int a = 0; a < MD_MAXTYPES; ++a) {
      if (t == a) {
        v[a] += d2;
        ++n[a];
      }
    }
  }
#pragma unroll
  for (int a = 0; a < MD_MAXTYPES; ++a) cnt[a] = (double)n[a];
  msd_reduce(v, cnt, ntypes, part + (int64_t)blockIdx.x * 2 * MD_MAXTYPES);
}

// The blocks' records, strided over the threads of one CTA, then as above.
__global__ void __launch_bounds__(MSD_THREADS) k_msd_final(int nblocks, int ntypes, const double* part, double* out) {
  __shared__ double tot[2 * MD_MAXTYPES];
  double v[MD_MAXTYPES] = {0, 0, 0, 0}, cnt[MD_MAXTYPES] = {0, 0, 0, 0};
  for (int t = threadIdx.x; t < nblocks; t += MSD_THREADS)
#pragma unroll
    for (int a = 0; a < MD_MAXTYPES; ++a)
      if (a < ntypes) {
        v[a] += part[(int64_t)t * 2 * MD_MAXTYPES + a];
        cnt[a] += part[(int64_t)t * 2 * MD_MAXTYPES + MD_MAXTYPES + a];
      }
  msd_reduce(v, cnt, ntypes, tot);
  __syncthreads();
  if (threadIdx.x < ntypes) out[threadIdx.x] = tot[MD_MAXTYPES + threadIdx.x] > 0 ? tot[threadIdx.x] / tot[MD_MAXTYPES + threadIdx.x] : 0.0;
}

// Pair-distance histogram of Sec. "Radial distribution function with
// Python": every unordered pair with r < nbins*dr adds 2 (like) or 1 (unlike)
// to bin floor(r/dr) of its replica (integer counts; exact, order-free).
//
// A warp takes a unit, the particles of up to RDF_CELLS neighbouring cells of
// one row, and the half of the rows around theirs that makes each pair of rows
// meet once (of its own row, the slots after each particle's). Row members are
// read 32 at a time, one per lane, straight from the gather copy, and tested in
// FP32 against each particle of the unit; pairs within rmax (one in six to nine)
// wait in a queue until a full warp of them is binned. The bin follows from the
// FP32 distance unless that lies within its own error of a bin edge; such pairs
// (about three in a thousand at dr = 0.01) are binned from the exact positions in
// FP64. So the counts are those of the exact distances, and GB300's slow FP64
// unit, which computed every pair's difference, root and quotient before, has
// next to nothing to do. Cells are those of the last list build; every particle
// has moved less than half the outer skin since, so rows are reached out to
// rmax + skin. A replica with too few cells for that is one row of all its slots.
// k_rdf_units lists the units that hold particles: most cells of a dilute box or
// of a plane hold none, and walking them took 1.3 s for 1000 particles in a box
// of 1024 cells per edge, where the whole call now takes 87 us.
// 400 bins to 4 sigma at N = 10^6: 2.6 ms (27 ms in FP64 throughout). What bounds
// a large system is the tests' issue slots, one below 10^5 particles the chain of
// one unit; units of 4 cells were slower at every N: 20 000 particles 424 us
// (now 254), 10^6 2836 us (units of 1 cell 3232).
#define RDF_SMEM_BINS 1024
#define RDF_CELLS 2
#define RDF_PART 16  // particles of a unit that are tested in one go
#define RDF_WARPS 8
// pairs that a warp bins before it moves the CTA's 32-bit counts to the 64-bit
// histogram (at N = 10^6 and 4 sigma it bins about 16 000 in all), and candidates
// between two looks at that number: a count stays below 2 RDF_WARPS (RDF_FLUSH +
// RDF_PART RDF_LOOK), 2.7e8, however large the system
#define RDF_FLUSH 65536
#define RDF_LOOK 1048576
// slots at whose multiples units are cut, so that no warp takes much more than
// this many particles, however many a cell holds (a droplet in a box of 1024
// wide cells per edge)
#define RDF_CUT 256
struct RdfArgs {
  bool mixed;
  int64_t ntot;
  int nbins, ndim, nrep;
  double dr, skin, iunit;  // (iunit: 1 / md_system::unit)
  const RepDev* reps;
  const int32_t* tile_rep;
  const uint4* xbq;   // positions at the last list build: the cells that slots are sorted by
  int32_t* unit;      // first slots of the units, replica r's from unit[off]
  int32_t* nunits;    // per replica
  int32_t* nowhere;   // per replica: whether a particle's position is NaN (FP64; its words are those of some place)
  const int32_t* blk; // first CTA of each replica, and the number of CTAs (one replica: not read)
  const uint4* pq;
  const uint64_t* pfx;
  const double4_32a* p4;
  const int32_t* cstart;
  unsigned long long* hist;
};
struct RdfWarp {
  float4 pos[RDF_PART];  // relative x, y, z, or words; the particle's type in w
  float r2[64];          // queue: squared distance, the other's slot, particle of the unit | class << 8
  int j[64];
  int c[64];
};

// The CTA's counts so far, moved by one warp: the exchange leaves the other
// warps free to go on counting.
__device__ __forceinline__ void rdf_flush(unsigned int* sh_h, int n, unsigned long long* h) {
  __syncwarp();
  for (int t = threadIdx.x & 31; t < n; t += 32) {
    const unsigned int v = atomicExch(&sh_h[t], 0u);
    if (v) atomicAdd(&h[t], (unsigned long long)v);
  }
  __syncwarp();
}

template <bool REL>
__device__ __forceinline__ void rdf_scan(const RdfArgs& a, const RepDev& R, RdfWarp& W, unsigned int* sh_h, bool priv, int r,
                                         int i0, int np, uint4 ref, int lo, int n, bool own, float rmax2f, float invdr,
                                         float edge, int& head, int& count) {
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const float sc = R.fxs;
  auto bin = [&](int m) {  // the first m queued pairs
    __syncwarp();
    if (lane < m) {
      const int q = (head + lane) & 63;
      const float t = sqrtf(W.r2[q]) * invdr, fl = floorf(t);
      const int cls = W.c[q] >> 8;
      int k = (int)fl;
      if (t - fl < edge || t - fl > 1.0f - edge) {
        const int64_t i = i0 + (W.c[q] & 255), j = W.j[q];
        const double rmax = a.dr * a.nbins;
        double d[3];
        for (int c = 0; c < 3; ++c) {
          if (a.mixed) {
            d[c] = (double)(int64_t)(a.pfx[c * a.ntot + i] - a.pfx[c * a.ntot + j]) * (R.L * (1.0 / 18446744073709551616.0));
          } else {
            const double xi = c == 0 ? a.p4[i].x : c == 1 ? a.p4[i].y : a.p4[i].z;
            const double xj = c == 0 ? a.p4[j].x : c == 1 ? a.p4[j].y : a.p4[j].z;
            double e = xi - xj;
            if (e > 0.5 * R.L) e -= R.L;
            else if (e < -0.5 * R.L) e += R.L;
            d[c] = e;
          }
        }
        const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
        k = r2 < rmax * rmax ? (int)(sqrt(r2) / a.dr) : a.nbins;
      }
      if (k < a.nbins) {
        const int slot = cls * a.nbins + k;
        const unsigned w = cls < 2 ? 2u : 1u;
        if (priv) atomicAdd(&sh_h[slot], w);
        else atomicAdd(&a.hist[(int64_t)r * 3 * a.nbins + slot], (unsigned long long)w);
      }
    }
    __syncwarp();
    head += m;
    count -= m;
  };
  if (lo < 0) {  // the unit is done: bin what waits
    if (count > 0) bin(count);
    return;
  }
  for (int t0 = 0; t0 < n; t0 += 32) {
    const int j = lo + t0 + lane;
    const bool in = t0 + lane < n;
    uint4 q = make_uint4(0u, 0u, 0u, 0u);
    if (in) q = a.pq[j];
    float x = 0.f, y = 0.f, z = 0.f;
    if (REL) {
      x = (float)(int)(q.x - ref.x) * sc;
      y = (float)(int)(q.y - ref.y) * sc;
      z = (float)(int)(q.z - ref.z) * sc;
    }
#pragma unroll 4
    for (int k = 0; k < np; ++k) {
      const float4 P = W.pos[k];
      float dx, dy, dz;
      if (REL) {
        dx = P.x - x;
        dy = P.y - y;
        dz = P.z - z;
      } else {
        dx = (float)(int)(__float_as_uint(P.x) - q.x) * sc;
        dy = (float)(int)(__float_as_uint(P.y) - q.y) * sc;
        dz = (float)(int)(__float_as_uint(P.z) - q.z) * sc;
      }
      const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
      const bool hit = in & (r2 < rmax2f) & (!own | (j > i0 + k));
      const unsigned m = __ballot_sync(0xffffffffu, hit);
      if (m == 0u) continue;
      if (hit) {
        const int e = (head + count + __popc(m & below)) & 63;
        const int ti = __float_as_int(P.w), tj = (int)q.w;
        W.r2[e] = r2;
        W.j[e] = j;
        W.c[e] = k | ((ti == tj ? ti : 2) << 8);
      }
      count += __popc(m);
      if (count >= 32) bin(32);
    }
  }
}

// Layers of cells that hold the partners within reach (rmax + skin); false: too few cells for
// that, every slot of the replica is a candidate.
__device__ __host__ __forceinline__ bool rdf_layers(double reach, int nc, float cellw, int* layers) {
  *layers = nc > 0 ? (int)ceil(reach * (1.0 + 1e-6) / (double)cellw) : 0;
  return nc > 0 && 2 * *layers + 1 <= nc;
}

// Cell of a slot at the last list build (the binning that sorted the slots).
__device__ __forceinline__ int3 rdf_cell(const uint4& x, int nc) {
  return make_int3((int)(((uint64_t)x.x * (uint64_t)nc) >> 32), (int)(((uint64_t)x.y * (uint64_t)nc) >> 32),
                   (int)(((uint64_t)x.z * (uint64_t)nc) >> 32));
}

// First slots of the units. A warp is a tile; the CTA's units of a replica are
// listed together and in order, so that the warps of a CTA of k_rdf work side by
// side and share rows in L1 (the order of the CTAs is left open: counts do not
// depend on it).
#define RDF_LIST 1024
__global__ void __launch_bounds__(RDF_LIST) k_rdf_units(RdfArgs a) {
  __shared__ int sh_r[RDF_LIST / 32], sh_n[RDF_LIST / 32], sh_base[RDF_LIST / 32];
  const int64_t i = (int64_t)blockIdx.x * RDF_LIST + threadIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool in = i < a.ntot;
  const int r = in ? a.tile_rep[i >> 5] : -1;
  const RepDev& R = a.reps[in ? r : 0];
  const int64_t k = i - R.off;
  bool first = false;
  int layers;
  if (in && k < R.n) {
    if (!a.mixed) {
      const double4_32a x = a.p4[i];
      if (isnan(x.x) || isnan(x.y) || isnan(x.z)) a.nowhere[r] = 1;
    }
    if (!rdf_layers((a.dr * a.nbins + a.skin) * a.iunit, R.nc, R.cellw, &layers)) {
      first = k % RDF_PART == 0;
    } else if (k == 0 || i % RDF_CUT == 0) {
      first = true;
    } else {
      const int3 c = rdf_cell(a.xbq[i], R.nc), d = rdf_cell(a.xbq[i - 1], R.nc);
      first = c.x / RDF_CELLS != d.x / RDF_CELLS || c.y != d.y || c.z != d.z;
    }
  }
  const unsigned m = __ballot_sync(0xffffffffu, first);
  if (lane == 0) {
    sh_r[warp] = r;
    sh_n[warp] = __popc(m);
  }
  __syncthreads();
  // the tiles of this one's replica: units in those before it, and in all
  const bool same = sh_r[lane] == r;
  const unsigned tiles = __ballot_sync(0xffffffffu, same);
  const int before = __reduce_add_sync(0xffffffffu, same && lane < warp ? sh_n[lane] : 0);
  const int all = __reduce_add_sync(0xffffffffu, same ? sh_n[lane] : 0);
  const int head = __ffs(tiles) - 1;
  if (warp == head && lane == 0 && in) sh_base[warp] = atomicAdd(&a.nunits[r], all);
  __syncthreads();
  if (first) a.unit[R.off + sh_base[head] + before + __popc(m & ((1u << lane) - 1u))] = (int32_t)i;
}

__global__ void __launch_bounds__(32 * RDF_WARPS) k_rdf(RdfArgs a) {
  __shared__ unsigned int sh_h[3 * RDF_SMEM_BINS];
  __shared__ RdfWarp sh_w[RDF_WARPS];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int r = 0, b = blockIdx.x, nblk = gridDim.x;
  if (a.nrep > 1) {
    int hi = a.nrep;  // blk[r] <= blockIdx.x < blk[hi]
    while (hi - r > 1) {
      const int mid = (r + hi) >> 1;
      if (a.blk[mid] <= b) r = mid; else hi = mid;
    }
    nblk = a.blk[r + 1] - a.blk[r];
    b -= a.blk[r];
  }
  const RepDev& R = a.reps[r];
  const bool priv = a.nbins <= RDF_SMEM_BINS;
  if (priv)
    for (int t = threadIdx.x; t < 3 * a.nbins; t += blockDim.x) sh_h[t] = 0u;
  __syncthreads();
  const double dr = a.dr * a.iunit, rmax = dr * a.nbins;  // as the FP32 numbers are
  const int nc = R.nc;
  int layers;
  const bool all = !rdf_layers(rmax + a.skin * a.iunit, nc, R.cellw, &layers);
  const int units = a.nunits[r];
  const bool rel = !all && 2 * (RDF_CELLS + layers + 1) < nc;
  // the FP32 distance is off by less than err: the rounding of coordinates of
  // at most `span`, and the words' own error
  const double span = rel ? (double)(RDF_CELLS + layers + 1) * (double)R.cellw : rmax;
  const double err = 1e-6 * span + 8.0 * (R.L * a.iunit) / 4294967296.0;
  // (with a particle that is nowhere every pair is binned from the exact positions)
  const float edge = a.nowhere[r] ? 1.0f : (float)(err / dr + 1e-6 * a.nbins), invdr = (float)(1.0 / dr);
  const float rmax2f = (float)((rmax + 2.0 * err) * (rmax + 2.0 * err) * (1.0 + 1e-6));
  RdfWarp& W = sh_w[warp];
  int head = 0, count = 0;  // the queue; head also counts the pairs binned since the last flush
  for (int64_t u = b * RDF_WARPS + warp; u < units; u += (int64_t)nblk * RDF_WARPS) {
    const int s0 = a.unit[R.off + u];
    int s1, x0 = 0, cy = 0, cz = 0, g = 0;
    if (all) {
      s1 = min(s0 + RDF_PART, (int)R.off + R.n);
    } else {
      const int3 c = rdf_cell(a.xbq[s0], nc);
      x0 = c.x / RDF_CELLS * RDF_CELLS;
      cy = c.y;
      cz = c.z;
      g = min(RDF_CELLS, nc - x0);
      s1 = min(a.cstart[R.cs0 + (cz * nc + cy) * nc + x0 + g], s0 / RDF_CUT * RDF_CUT + RDF_CUT);
    }
    for (int i0 = s0; i0 < s1; i0 += RDF_PART) {
      const int np = min(RDF_PART, s1 - i0);
      const uint4 ref = a.pq[i0];
      __syncwarp();
      if (lane < np) {
        const uint4 q = a.pq[i0 + lane];
        const float t = __int_as_float((int)q.w);
        W.pos[lane] = rel ? make_float4((float)(int)(q.x - ref.x) * R.fxs, (float)(int)(q.y - ref.y) * R.fxs,
                                        (float)(int)(q.z - ref.z) * R.fxs, t)
                          : make_float4(__uint_as_float(q.x), __uint_as_float(q.y), __uint_as_float(q.z), t);
      }
      __syncwarp();
      auto scan = [&](int lo, int n, bool own) {
        do {
          const int m = min(n, RDF_LOOK);
          if (rel) rdf_scan<true>(a, R, W, sh_h, priv, r, i0, np, ref, lo, m, own, rmax2f, invdr, edge, head, count);
          else rdf_scan<false>(a, R, W, sh_h, priv, r, i0, np, ref, lo, m, own, rmax2f, invdr, edge, head, count);
          if (head >= RDF_FLUSH) {
            if (priv) rdf_flush(sh_h, 3 * a.nbins, a.hist + (int64_t)r * 3 * a.nbins);
            head &= 63;
          }
          lo += m;
          n -= m;
        } while (n > 0);
      };
      if (all) {
        scan(i0, (int)R.off + R.n - i0, true);
      } else {
        const int len = min(2 * layers + g, nc);
        const int a0 = len == nc ? 0 : (x0 - layers + nc) % nc;
        const int over = max(a0 + len - nc, 0);
        // rows (oy, oz): (0..layers, 0), then (-layers..layers, 1..layers); their
        // runs [a0, a0 + len) of cells, in two parts where they pass the box
        // edge, are looked up by one lane each
        const int wide = 2 * layers + 1;
        const int rows = layers + 1 + (a.ndim == 3 ? layers * wide : 0);
        for (int q0 = 0; q0 < rows; q0 += 32) {
          const int q = q0 + lane;
          int lo0 = 0, n0 = 0, lo1 = 0, n1 = 0;
          if (q < rows) {
            const int oz = q <= layers ? 0 : 1 + (q - layers - 1) / wide;
            const int oy = q <= layers ? q : (q - layers - 1) % wide - layers;
            const int32_t* cs = a.cstart + R.cs0 + (((cz + oz) % nc) * nc + (cy + oy + nc) % nc) * nc;
            lo0 = cs[a0];
            n0 = cs[a0 + len - over] - lo0;
            if (over > 0) {
              lo1 = cs[0];
              n1 = cs[over] - lo1;
            }
          }
          for (int part = 0; part < 2; ++part)
            for (unsigned m = __ballot_sync(0xffffffffu, (part ? n1 : n0) > 0); m; m &= m - 1u) {
              const int from = __ffs(m) - 1;
              scan(__shfl_sync(0xffffffffu, part ? lo1 : lo0, from), __shfl_sync(0xffffffffu, part ? n1 : n0, from),
                   q0 + from == 0);
            }
        }
      }
      scan(-1, 0, false);
    }
  }
  if (!priv) return;
  __syncthreads();
  unsigned long long* h = a.hist + (int64_t)r * 3 * a.nbins;
  for (int t = threadIdx.x; t < 3 * a.nbins; t += blockDim.x)
    if (sh_h[t]) atomicAdd(&h[t], (unsigned long long)sh_h[t]);
}

// Pairs (i < j) inside their cutoff r < r_c,ab, from exact distances (mixed:
// 64-bit fixed-point differences; FP64: the minimum-image branch rule), found
// through the cells of the last list build. Every particle has moved less
// than half the outer skin since, so the cells within (r_c,max + skin_outer)
// of its current position hold every partner; a replica with too few cells
// for that is scanned whole.
__global__ void k_count_pairs(bool mixed, int64_t ntot, int ntypes, double reach, const RepDev* reps,
                              const int32_t* tile_rep, const uint64_t* pfx, const double4_32a* p4, const uint8_t* typ,
                              const int32_t* cstart, const double* rc2d, unsigned long long* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ntot) return;
  const RepDev& R = reps[tile_rep[i >> 5]];
  if (i - R.off >= R.n) return;
  const int ti = typ[i];
  double xi[3];
  uint64_t ui[3];
  for (int c = 0; c < 3; ++c) {
    if (mixed) ui[c] = pfx[c * ntot + i];
    else xi[c] = c == 0 ? p4[i].x : c == 1 ? p4[i].y : p4[i].z;
  }
  unsigned long long cnt = 0;
  auto visit = [&](int64_t j) {
    if (j <= i) return;
    double d2 = 0.0;
    for (int c = 0; c < 3; ++c) {
      double d;
      if (mixed) {
        d = (double)(int64_t)(ui[c] - pfx[c * ntot + j]) * (R.L * (1.0 / 18446744073709551616.0));
      } else {
        const double xj = c == 0 ? p4[j].x : c == 1 ? p4[j].y : p4[j].z;
        d = xi[c] - xj;
        if (d > 0.5 * R.L) d -= R.L;
        else if (d < -0.5 * R.L) d += R.L;
      }
      d2 += d * d;
    }
    cnt += d2 < rc2d[ti * ntypes + typ[j]];
  };
  const int nc = R.nc;
  const int layers = nc > 0 ? (int)ceil(reach * (1.0 + 1e-6) / (double)R.cellw) : 0;
  if (nc == 0 || 2 * layers + 1 > nc) {
    for (int64_t j = R.off; j < R.off + R.n; ++j) visit(j);
  } else {
    int cc[3];
    for (int c = 0; c < 3; ++c) {
      if (mixed) cc[c] = (int)(((uint64_t)(uint32_t)(ui[c] >> 32) * (uint64_t)nc) >> 32);
      else cc[c] = min(max((int)(xi[c] * (double)nc * R.invL), 0), nc - 1);
    }
    for (int oz = -layers; oz <= layers; ++oz)
      for (int oy = -layers; oy <= layers; ++oy)
        for (int ox = -layers; ox <= layers; ++ox) {
          const int c = (((cc[2] + oz + 8 * nc) % nc) * nc + (cc[1] + oy + 8 * nc) % nc) * nc + (cc[0] + ox + 8 * nc) % nc;
          for (int j = cstart[R.cs0 + c]; j < cstart[R.cs0 + c + 1]; ++j) visit(j);
        }
  }
  if (cnt) atomicAdd(out, cnt);
}

// Sum of n non-negative ints (warp sums, one atomic per warp).
__global__ void k_sum_i32(int64_t n, const int32_t* v, unsigned long long* out) {
  unsigned long long acc = 0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    acc += (unsigned long long)v[k];
  acc = kamd::warp_sum(acc);
  if ((threadIdx.x & 31) == 0 && acc) atomicAdd(out, acc);
}

int blocks_for(int64_t n, int b) { return (int)((n + b - 1) / b); }

// ------------------------------------------------------------------ host helpers

// The control block and the replicas live in one device allocation, so that
// one copy each way serves a launch. Only the persistent kernel changes them
// on the device: the host's mirrors are sent before a launch (the replicas
// only if the host changed them) and fetched after it, into pinned memory, and
// stay current until the next one. (A call used to make up to four copies to
// the host, each into pageable memory with a wait, and up to four to the
// device: FP64 forces of 1000 particles 210 -> 192 us, 50 Nose-Hoover steps of
// 1000 particles in a plane 931 -> 907 us, 100 steps of 32 000 from host
// arrays and back 2826 -> 2758 us.)
constexpr size_t CTL_BYTES = (sizeof(CtlDev) + 255) / 256 * 256;
// batches beyond this many replicas (0.4 MB) fetch the replicas only when a call needs them
constexpr int LAND_REPS = 1024;

md_status upload_reps(md_system* s) {
  CK(cudaMemcpyAsync(s->d_reps, s->reps.data(), sizeof(RepDev) * s->nrep, cudaMemcpyHostToDevice, s->stream));
  s->reps_dirty = false;
  return MD_OK;
}
md_status upload_state(md_system* s) {
  // (many replicas go by themselves: putting 1.6 MB of them together cost more than a second copy does)
  if (s->reps_dirty && s->nrep > LAND_REPS) CKS(upload_reps(s));
  const size_t nr = s->reps_dirty ? sizeof(RepDev) * (size_t)s->nrep : 0;
  const size_t bytes = CTL_BYTES + nr;
  if (s->up.size() < bytes) s->up.resize(bytes);
  std::memcpy(s->up.data(), &s->ctl, sizeof(CtlDev));
  if (nr) std::memcpy(s->up.data() + CTL_BYTES, s->reps.data(), nr);
  CK(cudaMemcpyAsync(s->d_state, s->up.data(), bytes, cudaMemcpyHostToDevice, s->stream));
  s->reps_dirty = false;
  return MD_OK;
}
md_status download_state(md_system* s, bool with_reps) {
  const bool reps = with_reps && !s->reps_now;
  if (s->ctl_now && !reps) return MD_OK;
  const size_t nr = sizeof(RepDev) * (size_t)s->nrep;
  const bool land = reps && s->nrep <= LAND_REPS;
  CK(cudaMemcpyAsync(s->h_land, s->d_state, land ? CTL_BYTES + nr : sizeof(CtlDev), cudaMemcpyDeviceToHost, s->stream));
  if (reps && !land) CK(cudaMemcpyAsync(s->reps.data(), s->d_reps, nr, cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  if (!s->ctl_now) std::memcpy(&s->ctl, s->h_land, sizeof(CtlDev));
  if (land) std::memcpy(s->reps.data(), s->h_land + CTL_BYTES, nr);
  s->ctl_now = true;
  if (reps) s->reps_now = true;
  return MD_OK;
}
md_status download_reps(md_system* s) { return download_state(s, true); }
md_status download_ctl(md_system* s) { return download_state(s, false); }

double rc_max(const md_system* s) {
  double m = 0;
  for (int t = 0; t < s->ntypes * s->ntypes; ++t) m = std::max(m, s->rc[t]);
  return m;
}

// Lanes per particle in the lists: the tuning's, but at least four on the FP64
// path, whose force phase costs what its FP64 instructions cost: units of eight
// particles spread them evenly over the SMs (N = 32 000: 26 units per SM
// instead of 6.6, which left the FP64 pipes 18 % idle).
int list_lanes(const md_system* s) { return s->mixed ? s->tun.threads_per_atom : std::max(4, s->tun.threads_per_atom); }

// Cells per edge and list capacity follow from the skin; both are recomputed
// whenever the tuning changes. Cells are at least half the outer list radius
// wide, so the list build scans the 5 x 5 x 5 cells around a particle's own
// (less volume than 27 cells of the full radius, and the corners are culled);
// a box with fewer than 8 such cells per edge uses cells of the full radius
// (3 x 3 x 3), and one with fewer than 3 of those an all-pairs scan.
// KAMD_CELL_REACH=1 keeps cells of the full radius (for tests of that path).
// Cells are wider than that by more than the 32-bit words, from which particles
// are binned, lie off the positions.
void layout_cells(md_system* s) {
  const double rl = rc_max(s) + s->tun.skin_outer;
  int reach = 2;
  if (const char* e = std::getenv("KAMD_CELL_REACH")) reach = std::atoi(e) == 1 ? 1 : 2;
  int64_t cell0 = 0;
  for (int r = 0; r < s->nrep; ++r) {
    RepDev& R = s->reps[r];
    int nr = reach;
    const double off = std::ldexp(R.L, -31);
    int nc = (int)std::min(std::floor(R.L / (rl / nr + off)), 1024.0);
    const int nc1 = (int)std::floor(R.L / (rl + off));
    // full-width cells where they fit 3 per edge and half-width cells fewer
    // than 8 (measured on 8 replicas of N = 1000, L = 9.41: 6 half-width
    // cells per edge were 13 % slower than 3 full-width ones), and where the
    // box is too small for 5 half-width cells; half-width cells otherwise
    // (N = 1000 with an outer radius of 3.7: 5 half-width cells per edge were
    // twice as fast as an all-pairs scan)
    if (nr == 2 && ((nc < 8 && nc1 >= 3) || nc < 5)) {
      nr = 1;
      nc = nc1;
    }
    if (nc < 3) nc = 0;
    R.nc = nc;
    R.nr = nc > 0 ? nr : 1;
    R.cellw = nc > 0 ? (float)(R.L / nc / s->unit) : 0.0f;
    // Margin of the FP64 path's squared distances from 32-bit words. Per coordinate,
    // a difference of words is off by off/2; the list build's differences of FP32
    // coordinates, up to four cells from the group's first particle, by another
    // 1.5 off in the widest cells (1024 per edge; in narrower ones the tests'
    // relative 1e-5 holds that); and two particles may each have moved off/2 more
    // than the triggers see: 3 off in all, taken as 4
    const double err = 4.0 * std::sqrt(3.0) * off / s->unit;
    R.mg = s->mixed ? 0.0f : (float)((2.0 * rl / s->unit + err) * err);
    R.cell0 = cell0;
    R.cs0 = cell0 + r;
    cell0 += (int64_t)nc * nc * nc;
  }
  s->ncells = cell0;
}

int list_capacity(const md_system* s) {
  const double rl = rc_max(s) + s->tun.skin_outer;
  double dens = 0;
  int64_t nmax = 0;
  for (int r = 0; r < s->nrep; ++r) {
    const double Lr = s->L_per[r];
    dens = std::max(dens, (double)s->n_per[r] / (s->ndim == 3 ? Lr * Lr * Lr : Lr * Lr));
    nmax = std::max(nmax, s->n_per[r]);
  }
  // particles within the list radius: a sphere, or in two dimensions a disc
  double est = s->ndim == 3 ? 4.0 / 3.0 * M_PI * rl * rl * rl * dens : M_PI * rl * rl * dens;
  int cap = (int)std::min(std::ceil(1.5 * est + 32), 1e9);  // (a skin may be many times the box)
  // KAMD_LIST_CAPACITY: start from a given capacity (the list still grows on overflow)
  if (const char* e = std::getenv("KAMD_LIST_CAPACITY")) cap = std::max(1, std::atoi(e));
  if (cap > nmax - 1) cap = (int)std::max<int64_t>(nmax - 1, 1);
  return cap;
}

// List-build groups, per replica: as many neighbouring cells per CTA (powers
// of two up to 4 x 4 x 4, 4 x 4 in a plane) as T threads per particle fill to
// at most 90 % of the CTA, from the replica's own cells (a batch can mix
// half-width, full-width and no cells). KAMD_LIST_GROUP forces one size.
void choose_groups(md_system* s) {
  const int gmax = s->ndim == 3 ? 64 : 16;
  int forced = 0;
  if (const char* e = std::getenv("KAMD_LIST_GROUP")) {
    const int v = std::atoi(e);
    if (v >= 1 && v <= gmax && (v & (v - 1)) == 0) forced = v;
  }
  for (int r = 0; r < s->nrep; ++r) {
    RepDev& R = s->reps[r];
    int g = 1;
    if (R.nc > 0) {
      // particles per occupied cell (two dimensions: only the cells of the plane hold particles)
      const double w = (double)R.cellw * s->unit;
      const double occ = s->ndim == 3 ? (double)s->n_per[r] / (R.L * R.L * R.L) * w * w * w
                                      : (double)s->n_per[r] / (R.L * R.L) * w * w;
      // 10 % headroom: a group whose particles overflow the CTA needs a second,
      // mostly idle pass (measured: 1.7x slower list build at N = 32 000, T = 2).
      // Groups stop at 64 cells: the staging area of 128-cell groups (57 KB per
      // CTA at N = 10^6) takes shared memory from the L1 cache that the force
      // phase's gathers use (list build 20 % faster, force phase 8 % slower)
      const double fit = 0.9 * (double)s->tun.block_size / ((double)list_lanes(s) * occ);
      while (2 * g <= gmax && 2 * g <= fit) g *= 2;
    }
    if (forced) g = forced;
    // x doubles first, then y, then z (a plane: x and y only)
    int gx = 1, gy = 1, gz = 1;
    for (int k = 1; k < g; k *= 2) {
      if (gx <= gy && (s->ndim == 2 || gx <= gz) && gx < 4) gx *= 2;
      else if (gy <= gz || s->ndim == 2) gy *= 2;
      else gz *= 2;
    }
    R.gx = gx;
    R.gy = gy;
    R.gz = gz;
    R.ngrp = R.nc > 0 ? ((R.nc + gx - 1) / gx) * ((R.nc + gy - 1) / gy) * ((R.nc + gz - 1) / gz) : 1;
  }
}

// Staging area of the list build: the candidates of the cells around one
// group, (gx+2)(gy+2)(gz+2) cells (or a whole replica too small for cells),
// with headroom over the mean (overflow regrows it).
int stage_capacity(md_system* s) {
  choose_groups(s);
  int cap = 64;
  for (int r = 0; r < s->nrep; ++r) {
    const RepDev& R = s->reps[r];
    // occupied union cells (two dimensions: one plane of cells)
    const int e = 2 * R.nr;
    const double nu = s->ndim == 3 ? (double)(R.gx + e) * (R.gy + e) * (R.gz + e) : (double)(R.gx + e) * (R.gy + e);
    const double w = (double)R.cellw * s->unit;
    const double occ = s->ndim == 3 ? (double)s->n_per[r] / (R.L * R.L * R.L) * w * w * w
                                    : (double)s->n_per[r] / (R.L * R.L) * w * w;
    int need;
    if (R.nc > 0) {
      const double mean = nu * occ;
      need = (int)std::ceil(1.1 * mean + 6.0 * std::sqrt(mean) + 32.0);
    } else {
      need = (int)s->n_per[r];
    }
    cap = std::max(cap, need);
  }
  return cap;
}

// Dynamic shared memory of the persistent kernel: the list build's staging area;
// the FP64 path's force phase uses it for its queues (2 KB per warp).
size_t stage_bytes(const md_system* s) {
  const size_t stage = (size_t)s->stage_cap * 16;
  return s->mixed ? stage : std::max(stage, (size_t)s->tun.block_size / 32 * 2048);
}

md_status alloc_cells_and_list(md_system* s, int cap_entries) {
  const int T = list_lanes(s);
  dfree(s, s->d_ccount);
  dfree(s, s->d_cstart);
  dfree(s, s->d_ccursor);
  dfree(s, s->d_chunk);
  dfree(s, s->d_nbr);
  dfree(s, s->d_nbr_in);
  dfree(s, s->d_cell_rep);
  s->maxrows = ((cap_entries + T - 1) / T + 3) / 4 * 4;  // list layout: whole quads per column
  CKS(dalloc(s, &s->d_cell_rep, (size_t)s->ncells));
  {
    std::vector<int32_t> cr((size_t)std::max<int64_t>(s->ncells, 1), 0);
    for (int r = 0; r < s->nrep; ++r) {
      const int64_t nc3 = (int64_t)s->reps[r].nc * s->reps[r].nc * s->reps[r].nc;
      for (int64_t c = 0; c < nc3; ++c) cr[s->reps[r].cell0 + c] = r;
    }
    // on the system's stream, after dalloc's clearing memset; cr is a local vector
    CK(cudaMemcpyAsync(s->d_cell_rep, cr.data(), 4 * cr.size(), cudaMemcpyHostToDevice, s->stream));
    CK(cudaStreamSynchronize(s->stream));
  }
  CKS(dalloc(s, &s->d_ccount, (size_t)s->ncells));
  CKS(dalloc(s, &s->d_cstart, (size_t)(s->ncells + s->nrep)));
  CKS(dalloc(s, &s->d_ccursor, (size_t)s->ncells));
  CKS(dalloc(s, &s->d_chunk, (size_t)(s->ncells / MD_SCAN_CHUNK + 1)));
  {
    // two-level reductions (chunks of red_tiles tiles) once a replica spans
    // more than 4 chunks: below that, one CTA per replica is as fast and, in
    // NVE, its reduction overlaps the next step instead of adding a barrier.
    // KAMD_RED_TILES sets the chunk and the threshold to the same value, for
    // tests of that path.
    s->red_tiles = MD_RED_TILES;
    int threshold = 4 * MD_RED_TILES;
    if (const char* e = std::getenv("KAMD_RED_TILES")) {
      const int v = std::atoi(e);
      if (v >= 1) s->red_tiles = threshold = v;
    }
    std::vector<int2> rmap, rrep;
    int maxtiles = 0;
    for (int r = 0; r < s->nrep; ++r) {
      const int nch = (s->reps[r].ntiles + s->red_tiles - 1) / s->red_tiles;
      rrep.push_back(make_int2((int)rmap.size(), nch));
      for (int c = 0; c < nch; ++c) rmap.push_back(make_int2(r, c));
      maxtiles = std::max(maxtiles, s->reps[r].ntiles);
    }
    s->red2 = maxtiles > threshold ? 1 : 0;
    s->nred = (int64_t)rmap.size();
    dfree(s, s->d_redmap);
    dfree(s, s->d_redrep);
    dfree(s, s->d_redpart);
    s->d_redmap = nullptr;
    s->d_redrep = nullptr;
    s->d_redpart = nullptr;
    CKS(dalloc(s, &s->d_redmap, std::max<size_t>(rmap.size(), 1)));
    CKS(dalloc(s, &s->d_redrep, std::max<size_t>(rrep.size(), 1)));
    CKS(dalloc(s, &s->d_redpart, std::max<size_t>(rmap.size(), 1) * MD_NPART));
    if (!rmap.empty()) {
      CK(cudaMemcpyAsync(s->d_redmap, rmap.data(), sizeof(int2) * rmap.size(), cudaMemcpyHostToDevice, s->stream));
      CK(cudaMemcpyAsync(s->d_redrep, rrep.data(), sizeof(int2) * rrep.size(), cudaMemcpyHostToDevice, s->stream));
      CK(cudaStreamSynchronize(s->stream));  // local vectors
    }
  }
  const size_t entries = (size_t)s->ntiles * s->maxrows * 32 * T;
  CKS(dalloc(s, &s->d_nbr, entries));
  CKS(dalloc(s, &s->d_nbr_in, entries));
  s->list_bytes = entries * 8;
  return MD_OK;
}

md_status mark_rebuild_all(md_system* s) {
  CKS(download_reps(s));
  for (auto& R : s->reps) R.want_rebuild = 1;
  s->reps_dirty = true;
  CKS(download_ctl(s));
  s->ctl.pending |= MD_FLAG_REBUILD;
  return MD_OK;
}

md_status configure_grid(md_system* s) {
  const int b = s->tun.block_size;
  int per_sm = 0;
  if (stage_bytes(s) > 200 * 1024) return fail(s, MD_ERR_NLIST_OVERFLOW, "list-build staging exceeds shared memory");
  CK(md_occupancy(s->mixed, b, stage_bytes(s), &per_sm));
  if (per_sm < 1) return fail(s, MD_ERR_INVALID_ARG, "block size too large for the persistent kernel");
  // One CTA per SM where that holds all the work at once: every warp unit of the
  // force phase, and every group of a replica's list build on a CTA of its own
  // (replicas seldom rebuild together). Further CTAs would only take part in the
  // barriers. (One CTA per SM against two, T = 8 and 512 threads: N = 4000, 125
  // groups, force phase 5.8 -> 5.4 us, FP64 24.7 -> 23.1, list build 35 -> 29;
  // N = 9500, 216 groups, 6.6 -> 6.1 but list build 37 -> 54.)
  int groups = 0;
  for (const auto& R : s->reps) groups = std::max(groups, R.ngrp);
  const bool small = groups <= s->nsm && (int64_t)s->ntiles * list_lanes(s) <= (int64_t)s->nsm * (b / 32);
  for (int w = 0; w < 2; ++w) {
    const int n = w == 0 && small ? 1 : per_sm;
    s->shape[w].grid = n * s->nsm;
    // The split between shared memory and L1 is asked for at each launch: no more
    // shared memory than the resident CTAs take, since the force phase's gathers
    // live in L1. The driver's own choice was larger: N = 10^6, force phase 199 ->
    // 191 us; 20 steps of N = 8*10^6 56.3 -> 54.0 ms. (A launch attribute: other
    // systems of the process have other needs.)
    CK(md_carveout(s->mixed, stage_bytes(s), n, &s->shape[w].carveout));
  }
  const int most = s->shape[1].grid;
  if (most > s->cta_sm_cap) {
    dfree(s, s->d_cta_sm);
    s->d_cta_sm = nullptr;
    s->cta_sm_cap = 0;
    CKS(dalloc(s, &s->d_cta_sm, (size_t)most));
    s->cta_sm_cap = most;
  }
  return MD_OK;
}

void fill_tables(const md_system* s, KParams& p) {
  const int nt = s->ntypes;
  for (int t = 0; t < nt * nt; ++t) {
    const double e = s->eps[t], sg = s->sig[t], rc = s->rc[t];
    const double sr6 = std::pow(sg / rc, 6.0);
    const double vc = 4.0 * e * (sr6 * sr6 - sr6);
    const double u = s->unit;
    const double rl = (rc + s->tun.skin_outer) / u, rli = (rc + s->tun.skin) / u;
    const double sgu = sg / u, s6 = sgu * sgu * sgu * sgu * sgu * sgu;
    p.tab_d[t][0] = rc * rc;
    p.tab_d[t][1] = 48.0 * e * s6 * s6;
    p.tab_d[t][2] = 24.0 * e * s6;
    p.tab_d[t][3] = vc;
    p.tabe_d[t][0] = 4.0 * e * s6 * s6;
    p.tabe_d[t][1] = 4.0 * e * s6;
    p.rli2_f[t] = (float)(rli * rli * (1.0 + 1e-5));
    p.rcw2_f[t] = (float)((rc / u) * (rc / u) * (1.0 + 1e-5));
    p.tab_f[t][0] = (float)(rc * rc);
    p.tab_f[t][1] = (float)(sg * sg);
    p.tab_f[t][2] = (float)(48.0 * e);
    p.tab_f[t][3] = (float)(4.0 * e);
    p.vsh_f[t] = (float)vc;
    // the list tests run in FP32 on cell-relative coordinates: widen the
    // radius by a relative 1e-5 so rounding can never drop a pair at the edge
    p.rl2_f[t] = (float)(rl * rl * (1.0 + 1e-5));
  }
}

KParams make_params(const md_system* s) {
  KParams p;
  std::memset(&p, 0, sizeof(p));
  p.nrep = s->nrep;
  p.ntypes = s->ntypes;
  p.ndim = s->ndim;
  p.ntot = s->ntot;
  p.ntiles = s->ntiles;
  p.T = list_lanes(s);
  p.maxrows = s->maxrows;
  fill_tables(s, p);
  p.mass = s->mass;
  p.inv_mass = 1.0 / s->mass;
  // rebuild the outer list once a particle moved (skin_outer - skin)/2 since
  // its build (every pair within r_c + skin is then still in it); prune the
  // inner list once a particle moved skin/2 since the last prune. With
  // skin_outer == skin there is one list: rebuilt at skin/2, never pruned,
  // and the force phase reads it directly
  const double so = s->tun.skin_outer / s->unit, si = s->tun.skin / s->unit;
  p.dual = s->tun.skin_outer > s->tun.skin ? 1 : 0;
  p.skin_half2f = (float)(p.dual ? 0.25 * (so - si) * (so - si) : 0.25 * si * si);
  p.prune_half2f = p.dual ? (float)(0.25 * si * si) : (float)HUGE_VAL;
  p.scaled = s->unit != 1.0 ? 1 : 0;
  p.unit2 = s->unit * s->unit;
  p.iunit2 = 1.0 / p.unit2;
  p.massf = (float)s->mass;
  p.inv_massf = (float)(1.0 / s->mass);
  p.timeout_ns = s->timeout_ns;
  p.reps = s->d_reps;
  p.tile_rep = s->d_tile_rep;
  p.ctl = s->d_ctl;
  p.pfx = s->d_pfx;
  p.pq[0] = s->d_pq[0];
  p.pq[1] = s->d_pq[1];
  p.velf = s->d_velf;
  p.frcf = s->d_frcf;
  p.xbq = s->d_xbq;
  p.xbq_in = s->d_xbq_in;
  p.p4[0] = s->d_p4[0];
  p.p4[1] = s->d_p4[1];
  p.veld = s->d_veld;
  p.frcd = s->d_frcd;
  p.gid = s->d_gid;
  p.typ = s->d_typ;
  p.img = s->d_img;
  p.t_pfx = s->d_tpfx;
  p.t_p4 = s->d_tp4;
  p.t_vel = s->d_tvel;
  p.t_frc = s->d_tfrc;
  p.t_gid = s->d_tgid;
  p.t_typ = s->d_ttyp;
  p.t_img = s->d_timg;
  p.cellof = s->d_cellof;
  p.cell_rep = s->d_cell_rep;
  p.ncells = s->ncells;
  p.stage_cap = s->stage_cap;
  p.ccount = s->d_ccount;
  p.cstart = s->d_cstart;
  p.ccursor = s->d_ccursor;
  p.chunk = s->d_chunk;
  p.cta_sm = s->d_cta_sm;
  p.red2 = s->red2;
  p.red_tiles = s->red_tiles;
  p.nred = s->nred;
  p.redmap = s->d_redmap;
  p.redrep = s->d_redrep;
  p.redpart = s->d_redpart;
  p.scat = s->d_scat;
  p.nbr = s->d_nbr;
  p.nnb = s->d_nnb;
  p.nbr_in = p.dual ? s->d_nbr_in : s->d_nbr;
  p.nnb_in = p.dual ? s->d_nnb_in : s->d_nnb;
  p.part[0] = s->d_part[0];
  p.part[1] = s->d_part[1];
  p.plog = s->d_plog;
  p.plog_rec = s->d_plog_rec;
  p.plog_stride = (int64_t)s->ntiles * p.T * MD_NPART;
  p.plog_slots = (s->plog_slots > 0 && (size_t)s->plog_slots * (size_t)p.plog_stride <= s->plog_cap) ? s->plog_slots : 0;
  return p;
}

void drop_graph(LaunchShape& h) {
  if (h.gexec) cudaGraphExecDestroy(h.gexec);
  if (h.graph) cudaGraphDestroy(h.graph);
  h.gexec = nullptr;
  h.graph = nullptr;
  h.gnode = nullptr;
}

// Whether a launch takes as many CTAs as fit although one per SM holds each
// replica's groups: when replicas that rebuild together have more groups than
// there are SMs, and the steps that follow are too few to repay the wait for
// them with cheaper barriers. Measured on 8 replicas of 1000 that all rebuild
// (216 groups), T = 4 and 256 threads, 152 CTAs against 608: forces 185 and 137
// us, NVE of 20 steps 525 and 488, of 40 1128 and 1140; Nose-Hoover of 20 682 and
// 644, of 50 1679 and 1727; resampling of 50 829 and 1027; FP64 on 456 CTAs,
// 10 steps 672 and 662, of 20 1310 and 1314.
bool wide_launch(const md_system* s, int op, int kind, int64_t nsteps) {
  if (s->shape[0].grid == s->shape[1].grid || !(s->ctl.pending & MD_FLAG_REBUILD)) return false;
  if (!s->reps_now && !s->reps_dirty) return false;  // not known here
  if (op == MD_OP_FORCE_REPEAT || op == MD_OP_LIST_REPEAT) return false;
  int64_t groups = 0;
  for (const auto& R : s->reps) groups += R.want_rebuild ? R.ngrp : 0;
  const int64_t few = s->mixed && kind != MD_KIND_RESAMPLE ? 24 : 10;
  return groups > s->shape[0].grid && (op != MD_OP_STEPS || nsteps <= few);
}

// Launch the persistent kernel. By default through an instantiated CUDA graph
// holding one cooperative kernel node (built once per launch shape, its
// parameters updated per call); a direct cooperative launch if the graph
// cannot be built or KAMD_NO_GRAPH is set.
cudaError_t launch_persistent(md_system* s, const KParams& p, LaunchShape& h) {
  const size_t smem = stage_bytes(s);
  const int block = s->tun.block_size;
  if (s->use_graph) {
    KParams pc = p;
    void* args[] = {(void*)&pc};
    cudaKernelNodeParams kp = {};
    kp.func = (void*)md_persistent_fn(s->mixed);
    kp.gridDim = dim3(h.grid);
    kp.blockDim = dim3(block);
    kp.sharedMemBytes = (unsigned)smem;
    kp.kernelParams = args;
    cudaError_t e = cudaSuccess;
    if (!h.gexec || h.g_grid != h.grid || h.g_block != block || h.g_smem != smem || h.g_carveout != h.carveout) {
      drop_graph(h);
      e = cudaFuncSetAttribute(kp.func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e == cudaSuccess) e = cudaGraphCreate(&h.graph, 0);
      if (e == cudaSuccess) e = cudaGraphAddKernelNode(&h.gnode, h.graph, nullptr, 0, &kp);
      if (e == cudaSuccess) {
        cudaKernelNodeAttrValue v = {};
        v.cooperative = 1;
        e = cudaGraphKernelNodeSetAttribute(h.gnode, cudaKernelNodeAttributeCooperative, &v);
        if (e == cudaSuccess) {
          cudaKernelNodeAttrValue c = {};
          c.sharedMemCarveout = (unsigned)h.carveout;
          e = cudaGraphKernelNodeSetAttribute(h.gnode, cudaKernelNodeAttributePreferredSharedMemoryCarveout, &c);
        }
      }
      if (e == cudaSuccess) e = cudaGraphInstantiate(&h.gexec, h.graph, 0);
      if (e == cudaSuccess) {
        h.g_grid = h.grid;
        h.g_block = block;
        h.g_smem = smem;
        h.g_carveout = h.carveout;
      }
    } else {
      e = cudaGraphExecKernelNodeSetParams(h.gexec, h.gnode, &kp);
    }
    if (e == cudaSuccess) e = cudaGraphLaunch(h.gexec, s->stream);
    if (e == cudaSuccess) {
      ++s->graph_launches;
      return cudaSuccess;
    }
    // the driver refused the graph: clear the error and launch directly from now on
    cudaGetLastError();
    drop_graph(h);
    s->use_graph = false;
  }
  return md_launch_persistent(s->mixed, p, h.grid, block, smem, h.carveout, s->stream);
}

// Run the persistent kernel for one operation, growing the neighbour list
// and relaunching when it overflows. *steps_out receives completed steps.
md_status run_op(md_system* s, int op, int kind, double dt, int64_t nsteps, int64_t nstep_boltz, uint64_t seed,
                 int64_t log_every, int64_t log_cap, int64_t* steps_out) {
  int64_t done = 0;
  for (int attempt = 0; attempt < 8; ++attempt) {
    // clear the barrier counter and any error flag of an earlier launch (the
    // host mirror is current: every launch ends with a download of it)
    s->ctl.pending &= MD_FLAG_REBUILD;
    s->ctl.err_where = 0;
    LaunchShape& shape = s->shape[wide_launch(s, op, kind, nsteps - done) ? 1 : 0];
    CKS(upload_state(s));
    KParams p = make_params(s);
    p.op = op;
    p.kind = kind;
    p.dt = dt;
    p.dtf = (float)dt;
    p.nsteps = nsteps - done;
    p.nstep_boltz = nstep_boltz;
    p.seed = seed;
    p.log_every = log_every;
    p.log_step0 = done;
    p.log_cap = log_cap;
    p.thermo = s->d_thermo;
    s->ctl_now = s->reps_now = false;
    CK(launch_persistent(s, p, shape));
    ++s->kernel_launches;
    CKS(download_state(s, s->nrep <= LAND_REPS));
    if (op == MD_OP_STEPS) done += s->ctl.steps_done;
    const int pend = s->ctl.pending;
    // log records whose sums the launch left in slots (before a relaunch reuses them)
    if (!(pend & MD_FLAG_TIMEOUT) && s->ctl.log_slots_used > 0) {
      CK(md_launch_log_records(s->mixed, p, s->ctl.log_slots_used, s->tun.block_size, s->stream));
      ++s->kernel_launches;
    }
    if (pend & MD_FLAG_TIMEOUT) {
      s->have_state = false;
      char buf[160];
      std::snprintf(buf, sizeof buf, "grid barrier timed out (phase %d); state is undefined, call md_set_state",
                    s->ctl.err_where);
      return fail(s, MD_ERR_TIMEOUT, buf);
    }
    if (pend & MD_FLAG_UNSTABLE) {
      if (steps_out) *steps_out = done;
      return fail(s, MD_ERR_UNSTABLE, "NaN/Inf state or a particle moved >= L/4 in one step");
    }
    if (pend & MD_FLAG_OVERFLOW) {
      // a list column or the build's staging area was too small: grow both
      const int cap = s->maxrows * list_lanes(s);
      CKS(alloc_cells_and_list(s, cap + cap / 2 + 16));
      s->stage_cap = std::min(s->stage_cap + s->stage_cap / 2, 200 * 1024 / 16);
      CKS(configure_grid(s));
      CKS(mark_rebuild_all(s));
      continue;
    }
    if (steps_out) *steps_out = done;
    return MD_OK;
  }
  return fail(s, MD_ERR_NLIST_OVERFLOW, "neighbour list kept overflowing after growing it 8 times");
}

md_status ensure_thermo(md_system* s, int64_t records) {
  if (records <= s->thermo_cap) return MD_OK;
  dfree(s, s->d_thermo);
  CKS(dalloc(s, &s->d_thermo, (size_t)records));
  s->thermo_cap = records;
  return MD_OK;
}

// Take the current unwrapped positions as the reference r(t_w) of one MSD
// slot (Eq. (msdtw)); slots other than 0 get their buffer on first use.
md_status reset_msd_ref(md_system* s, int slot = 0) {
  if (!s->d_msd_ref[slot]) CKS(dalloc(s, &s->d_msd_ref[slot], 3 * (size_t)s->n_total));
  const int b = 256;
  k_unwrapped<<<blocks_for(s->ntot, b), b, 0, s->stream>>>(s->mixed, s->ntot, s->d_reps, s->d_tile_rep, s->d_pfx,
                                                           s->d_p4[s->ctl.cur], s->d_gid, s->d_img,
                                                           s->d_msd_ref[slot]);
  CK(cudaGetLastError());
  s->msd_valid[slot] = true;
  return MD_OK;
}

md_status after_new_state(md_system* s) {
  CKS(download_reps(s));
  CK(cudaStreamSynchronize(s->stream));  // the caller's arrays have been read
  s->ctl = CtlDev{};
  s->ctl.pending = MD_FLAG_REBUILD;
  s->ctl.cur = 0;
  s->ctl.step = 0;
  s->ctl_now = true;
  for (auto& R : s->reps) {
    R.want_rebuild = 1;
    R.xi = R.g = R.lns = R.lns_next = R.xi_a = 0.0;
    R.xif = R.xiaf = 0.0f;
    R.prune_epoch = R.rebuild_epoch = -1;
  }
  s->reps_dirty = true;
  s->have_state = true;
  for (int k = 1; k < MD_MSD_SLOTS; ++k) s->msd_valid[k] = false;  // references of the old state
  CKS(reset_msd_ref(s));
  s->rdf_meas = 0;
  return MD_OK;
}

md_status set_state_impl(md_system* s, const double* pos, const double* vel, int on_device) {
  const double* dpos = pos;
  const double* dvel = vel;
  const size_t bytes = sizeof(double) * 3 * (size_t)s->n_total;
  if (!on_device) {
    CK(cudaMemcpyAsync(s->d_io, pos, bytes, cudaMemcpyHostToDevice, s->stream));
    dpos = s->d_io;
    if (vel) {
      CK(cudaMemcpyAsync(s->d_io + 3 * s->n_total, vel, bytes, cudaMemcpyHostToDevice, s->stream));
      dvel = s->d_io + 3 * s->n_total;
    }
  }
  const int b = 256;
  k_set_state<<<blocks_for(s->n_total, b), b, 0, s->stream>>>(
      s->mixed, s->ndim, s->n_total, s->ntot, s->d_reps, s->d_rep_of_caller, s->d_typ_caller, dpos, dvel, 0, s->d_pfx,
      s->d_pq[0], s->d_velf, s->d_frcf, s->d_xbq, s->d_p4[0], s->d_veld, s->d_frcd, s->d_gid, s->d_typ, s->d_img);
  CK(cudaGetLastError());
  CK(cudaMemsetAsync(s->d_nnb, 0, sizeof(int32_t) * 8 * (size_t)s->ntot, s->stream));
  CK(cudaMemsetAsync(s->d_nnb_in, 0, sizeof(int32_t) * 8 * (size_t)s->ntot, s->stream));
  return after_new_state(s);
}

md_status validate_table(int ntypes, const double* eps, const double* sigma, const double* rc, const double* L, int nrep,
                         double skin) {
  if (ntypes < 1 || ntypes > MD_MAXTYPES) return fail(nullptr, MD_ERR_INVALID_ARG, "ntypes must be in [1, 4]");
  if (!eps || !sigma || !rc) return fail(nullptr, MD_ERR_INVALID_ARG, "eps, sigma and rc tables are required");
  for (int a = 0; a < ntypes; ++a)
    for (int b = 0; b < ntypes; ++b) {
      const int t = a * ntypes + b, u = b * ntypes + a;
      if (!(eps[t] > 0) || !(sigma[t] > 0) || !(rc[t] > 0))
        return fail(nullptr, MD_ERR_INVALID_ARG, "eps, sigma and rc must be > 0");
      if (eps[t] != eps[u] || sigma[t] != sigma[u] || rc[t] != rc[u])
        return fail(nullptr, MD_ERR_INVALID_ARG, "eps, sigma and rc tables must be symmetric");
      for (int r = 0; r < nrep; ++r)
        if (!(rc[t] < 0.5 * L[r]))
          return fail(nullptr, MD_ERR_INVALID_ARG, "every cutoff must be < L/2 (unique minimum image)");
    }
  if (!(skin >= 0)) return fail(nullptr, MD_ERR_INVALID_ARG, "skin must be >= 0");
  return MD_OK;
}

md_status destroy_fail(md_system* s, md_status st) {
  g_create_err = s->err;
  md_destroy(s);
  return st;
}

md_status tuning_ok(md_system* s, const md_tuning* t) {
  const int T = t->threads_per_atom, b = t->block_size;
  if (!(T == 1 || T == 2 || T == 4 || T == 8)) return fail(s, MD_ERR_INVALID_ARG, "threads_per_atom must be 1, 2, 4 or 8");
  if (!(b == 128 || b == 256 || b == 512)) return fail(s, MD_ERR_INVALID_ARG, "block_size must be 128, 256 or 512");
  if (b < 32 * T) return fail(s, MD_ERR_INVALID_ARG, "block_size must hold at least one 32-particle tile");
  if (!(t->skin >= 0) || !(t->skin < 2.0)) return fail(s, MD_ERR_INVALID_ARG, "skin must be in [0, 2)");
  if (!(t->skin_outer >= t->skin) || !(t->skin_outer < 3.0))
    return fail(s, MD_ERR_INVALID_ARG, "skin_outer must be in [skin, 3)");
  for (int r = 0; r < s->nrep; ++r)
    if (!(rc_max(s) < 0.5 * s->L_per[r])) return fail(s, MD_ERR_INVALID_ARG, "cutoff must be < L/2");
  return MD_OK;
}

}  // namespace

void kamd_set_global_error(const std::string& msg) { g_create_err = msg; }

// ====================================================================== ABI

extern "C" {

md_status md_create_batch_dim(int ndim, int nrep, const int64_t* n_per, const double* L_per, const uint8_t* types,
                              int ntypes, const double* eps, const double* sigma, const double* rc, double mass,
                              double skin, md_precision prec, void* stream, md_system** out) {
  if (!out) return fail(nullptr, MD_ERR_INVALID_ARG, "out must not be NULL");
  *out = nullptr;
  if (ndim != 2 && ndim != 3) return fail(nullptr, MD_ERR_INVALID_ARG, "ndim must be 2 or 3");
  if (nrep < 1 || !n_per || !L_per || !types) return fail(nullptr, MD_ERR_INVALID_ARG, "nrep >= 1 and arrays required");
  if (prec != MD_PREC_FP64 && prec != MD_PREC_MIXED) return fail(nullptr, MD_ERR_INVALID_ARG, "unknown precision");
  if (!(mass > 0)) return fail(nullptr, MD_ERR_INVALID_ARG, "mass must be > 0");
  int64_t ntotal = 0, nslots = 0;
  for (int r = 0; r < nrep; ++r) {
    if (n_per[r] < 2) return fail(nullptr, MD_ERR_INVALID_ARG, "every replica needs n >= 2");
    if (!(L_per[r] > 0) || !std::isfinite(L_per[r])) return fail(nullptr, MD_ERR_INVALID_ARG, "box edge must be > 0");
    if (n_per[r] >= (int64_t)1 << 30) return fail(nullptr, MD_ERR_INVALID_ARG, "too many particles");
    ntotal += n_per[r];
    nslots += (n_per[r] + 31) / 32 * 32;
  }
  // slot indices share a 32-bit word with a 2-bit type in the list build
  if (nslots >= (int64_t)1 << 30) return fail(nullptr, MD_ERR_INVALID_ARG, "at most 2^30 - 1 slots (particles padded to tiles of 32 per replica)");
  CKS(validate_table(ntypes, eps, sigma, rc, L_per, nrep, skin));
  for (int64_t g = 0; g < ntotal; ++g)
    if (types[g] >= ntypes) return fail(nullptr, MD_ERR_INVALID_ARG, "type index out of range");

  md_system* s = new md_system();
  s->ndim = ndim;
  s->stream = (cudaStream_t)stream;
  s->nrep = nrep;
  s->ntypes = ntypes;
  s->n_total = ntotal;
  s->mixed = prec == MD_PREC_MIXED;
  s->mass = mass;
  s->tun.skin = skin;
  s->tun.skin_outer = skin + 0.4;
  for (int t = 0; t < ntypes * ntypes; ++t) {
    s->eps[t] = eps[t];
    s->sig[t] = sigma[t];
    s->rc[t] = rc[t];
  }
  if (!s->mixed) s->unit = length_unit(rc_max(s));
  if (const char* e = std::getenv("KAMD_BARRIER_TIMEOUT_MS")) s->timeout_ns = (unsigned long long)std::atoll(e) * 1000000ull;
  if (const char* e = std::getenv("KAMD_NO_GRAPH")) s->use_graph = !(e[0] == '1');
  if (const char* e = std::getenv("KAMD_LOG_NOW")) s->log_now = e[0] == '1';
  cudaError_t ce = cudaGetDevice(&s->device);
  if (ce != cudaSuccess) return destroy_fail(s, cuda_fail(s, ce, "cudaGetDevice"));
  int major = 0, minor = 0, coop = 0;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, s->device);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, s->device);
  cudaDeviceGetAttribute(&s->nsm, cudaDevAttrMultiProcessorCount, s->device);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, s->device);
  if (major != 10 || minor != 3 || !coop) {
    s->err = "this library is built for sm_103a (GB300) with cooperative launch";
    return destroy_fail(s, MD_ERR_NOT_SUPPORTED);
  }
  // replicas: slot ranges padded to whole 32-particle tiles
  s->n_per.assign(n_per, n_per + nrep);
  s->L_per.assign(L_per, L_per + nrep);
  s->reps.resize(nrep);
  std::vector<int32_t> tile_rep;
  std::vector<int32_t> rep_of(ntotal);
  int64_t off = 0, o0 = 0;
  for (int r = 0; r < nrep; ++r) {
    RepDev R;
    std::memset(&R, 0, sizeof(R));
    R.off = off;
    R.out0 = o0;
    R.n = (int32_t)n_per[r];
    R.ntiles = (int32_t)((n_per[r] + 31) / 32);
    R.tile0 = (int32_t)(off / 32);
    R.L = L_per[r];
    R.invL = 1.0 / L_per[r];
    R.fx64 = 18446744073709551616.0 / L_per[r];
    R.Lf = (float)L_per[r];
    R.fxs = (float)(L_per[r] / 4294967296.0 / s->unit);
    R.fx64f = (float)R.fx64;
    R.fx32f = (float)(4294967296.0 / L_per[r]);
    R.fx32 = 4294967296.0 / L_per[r];
    s->reps[r] = R;
    s->out0.push_back(o0);
    for (int t = 0; t < R.ntiles; ++t) tile_rep.push_back(r);
    int64_t n0 = 0;
    for (int64_t k = 0; k < n_per[r]; ++k) {
      rep_of[o0 + k] = r;
      n0 += types[o0 + k] == 0;
    }
    s->n_type0.push_back(n0);
    off += (int64_t)R.ntiles * 32;
    o0 += n_per[r];
  }
  s->ntot = off;
  s->ntiles = (int)(off / 32);
  layout_cells(s);
  md_status st;
  const size_t nt = (size_t)s->ntot;
#define AL(ptr, cnt)                                   \
  do {                                                 \
    st = dalloc(s, &(ptr), (cnt));                     \
    if (st != MD_OK) return destroy_fail(s, st);       \
  } while (0)
  AL(s->d_state, CTL_BYTES + sizeof(RepDev) * (size_t)nrep);
  s->d_ctl = reinterpret_cast<CtlDev*>(s->d_state);
  s->d_reps = reinterpret_cast<RepDev*>(s->d_state + CTL_BYTES);
  ce = cudaHostAlloc((void**)&s->h_land, CTL_BYTES + sizeof(RepDev) * (size_t)std::min(nrep, LAND_REPS), cudaHostAllocDefault);
  if (ce != cudaSuccess) return destroy_fail(s, cuda_fail(s, ce, "cudaHostAlloc"));
  AL(s->d_plog_rec, (size_t)MD_LOG_SLOTS);
  AL(s->d_tile_rep, (size_t)s->ntiles);
  AL(s->d_pq[0], nt);
  AL(s->d_pq[1], nt);
  AL(s->d_xbq, nt);
  AL(s->d_xbq_in, nt);
  if (s->mixed) {
    AL(s->d_pfx, 3 * nt);
    AL(s->d_velf, 3 * nt);
    AL(s->d_frcf, 3 * nt);
    AL(s->d_tpfx, 3 * nt);
    float* tv = nullptr;
    float* tf = nullptr;
    AL(tv, 3 * nt);
    AL(tf, 3 * nt);
    s->d_tvel = tv;
    s->d_tfrc = tf;
  } else {
    AL(s->d_p4[0], nt);
    AL(s->d_p4[1], nt);
    AL(s->d_veld, 3 * nt);
    AL(s->d_frcd, 3 * nt);
    AL(s->d_tp4, nt);
    double* tv = nullptr;
    double* tf = nullptr;
    AL(tv, 3 * nt);
    AL(tf, 3 * nt);
    s->d_tvel = tv;
    s->d_tfrc = tf;
  }
  AL(s->d_gid, nt);
  AL(s->d_typ, nt);
  AL(s->d_img, 3 * nt);
  AL(s->d_tgid, nt);
  AL(s->d_ttyp, nt);
  AL(s->d_timg, 3 * nt);
  AL(s->d_cellof, nt);
  AL(s->d_scat, nt);
  AL(s->d_nnb, 8 * nt);
  AL(s->d_nnb_in, 8 * nt);
  AL(s->d_part[0], (size_t)s->ntiles * 8 * MD_NPART);
  AL(s->d_part[1], (size_t)s->ntiles * 8 * MD_NPART);
  AL(s->d_typ_caller, (size_t)ntotal);
  AL(s->d_rep_of_caller, (size_t)ntotal);
  AL(s->d_msd_ref[0], 3 * (size_t)ntotal);
  AL(s->d_io, 6 * (size_t)ntotal);
  AL(s->d_io_i, 3 * (size_t)ntotal);
  AL(s->d_msd_part, (size_t)MSD_BLOCKS * 2 * MD_MAXTYPES);
  AL(s->d_count, 1);
#undef AL
  s->stage_cap = stage_capacity(s);
  st = alloc_cells_and_list(s, list_capacity(s));
  if (st != MD_OK) return destroy_fail(s, st);
  ce = cudaMemcpyAsync(s->d_tile_rep, tile_rep.data(), 4 * tile_rep.size(), cudaMemcpyHostToDevice, s->stream);
  if (ce == cudaSuccess)
    ce = cudaMemcpyAsync(s->d_rep_of_caller, rep_of.data(), 4 * rep_of.size(), cudaMemcpyHostToDevice, s->stream);
  if (ce == cudaSuccess) ce = cudaMemcpyAsync(s->d_typ_caller, types, (size_t)ntotal, cudaMemcpyHostToDevice, s->stream);
  if (ce != cudaSuccess) return destroy_fail(s, cuda_fail(s, ce, "cudaMemcpyAsync"));
  st = upload_reps(s);
  if (st == MD_OK) st = configure_grid(s);
  if (st != MD_OK) return destroy_fail(s, st);
  ce = cudaStreamSynchronize(s->stream);
  if (ce != cudaSuccess) return destroy_fail(s, cuda_fail(s, ce, "cudaStreamSynchronize"));
  *out = s;
  return MD_OK;
}

md_status md_create_batch(int nrep, const int64_t* n_per, const double* L_per, const uint8_t* types, int ntypes,
                          const double* eps, const double* sigma, const double* rc, double mass, double skin,
                          md_precision prec, void* stream, md_system** out) {
  return md_create_batch_dim(3, nrep, n_per, L_per, types, ntypes, eps, sigma, rc, mass, skin, prec, stream, out);
}

md_status md_create(int64_t n, const uint8_t* types, int ntypes, double L, const double* eps, const double* sigma,
                    const double* rc, double mass, double skin, md_precision prec, void* stream, md_system** out) {
  return md_create_batch_dim(3, 1, &n, &L, types, ntypes, eps, sigma, rc, mass, skin, prec, stream, out);
}

md_status md_set_state(md_system* s, const double* pos, const double* vel, int on_device) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!pos) return fail(s, MD_ERR_INVALID_ARG, "pos must not be NULL");
  return set_state_impl(s, pos, vel, on_device);
}

md_status md_get_state(md_system* s, double* pos, double* vel, int32_t* images, int on_device) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state: call md_set_state or md_init_lattice first");
  const size_t n3 = 3 * (size_t)s->n_total;
  double* dp = on_device ? pos : (pos ? s->d_io : nullptr);
  double* dv = on_device ? vel : (vel ? s->d_io + n3 : nullptr);
  int32_t* di = on_device ? images : (images ? s->d_io_i : nullptr);
  CKS(download_ctl(s));
  const int b = 256;
  k_get_state<<<blocks_for(s->ntot, b), b, 0, s->stream>>>(s->mixed, s->ntot, s->d_reps, s->d_tile_rep, s->ctl.cur,
                                                           s->d_pfx, s->d_velf, s->d_p4[s->ctl.cur], s->d_veld,
                                                           s->d_gid, s->d_img, dp, dv, di);
  CK(cudaGetLastError());
  if (!on_device) {
    if (pos) CK(cudaMemcpyAsync(pos, dp, 8 * n3, cudaMemcpyDeviceToHost, s->stream));
    if (vel) CK(cudaMemcpyAsync(vel, dv, 8 * n3, cudaMemcpyDeviceToHost, s->stream));
    if (images) CK(cudaMemcpyAsync(images, di, 4 * n3, cudaMemcpyDeviceToHost, s->stream));
  }
  CK(cudaStreamSynchronize(s->stream));
  return MD_OK;
}

md_status md_init_lattice(md_system* s, const double* T0, double jitter, uint64_t seed) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!T0) return fail(s, MD_ERR_INVALID_ARG, "T0 must not be NULL");
  if (!(jitter >= 0)) return fail(s, MD_ERR_INVALID_ARG, "jitter must be >= 0");
  for (int r = 0; r < s->nrep; ++r)
    if (!(T0[r] >= 0)) return fail(s, MD_ERR_INVALID_ARG, "T0 must be >= 0");
  const int b = 256;
  k_lattice<<<blocks_for(s->n_total, b), b, 0, s->stream>>>(s->ndim, s->n_total, s->d_reps, s->d_rep_of_caller,
                                                            jitter, seed, s->d_io);
  CK(cudaGetLastError());
  CKS(set_state_impl(s, s->d_io, nullptr, 1));
  CKS(download_reps(s));
  for (int r = 0; r < s->nrep; ++r) s->reps[r].T_target = T0[r];
  s->reps_dirty = true;
  CKS(run_op(s, MD_OP_INITVEL, MD_KIND_NVE, 0.0, 0, 0, seed, 0, 0, nullptr));
  return MD_OK;
}

md_status md_forces(md_system* s, double* f, double* pe, double* virial, int on_device) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state: call md_set_state or md_init_lattice first");
  CKS(run_op(s, MD_OP_FORCES, MD_KIND_NVE, 0.0, 0, 0, 0, 0, 0, nullptr));
  if (f) {
    double* df = on_device ? f : s->d_io;
    const int b = 256;
    k_get_forces<<<blocks_for(s->ntot, b), b, 0, s->stream>>>(s->mixed, s->ntot, s->d_reps, s->d_tile_rep, s->d_frcf,
                                                              s->d_frcd, s->d_gid, df);
    CK(cudaGetLastError());
    if (!on_device) CK(cudaMemcpyAsync(f, df, 24 * (size_t)s->n_total, cudaMemcpyDeviceToHost, s->stream));
  }
  CKS(download_reps(s));
  CK(cudaStreamSynchronize(s->stream));  // f is complete
  for (int r = 0; r < s->nrep; ++r) {
    if (pe) pe[r] = s->reps[r].pe;
    if (virial) virial[r] = s->reps[r].vir;
  }
  return MD_OK;
}

static md_status step_common(md_system* s, int kind, double dt, int64_t nsteps, int64_t nstep_boltz, uint64_t seed,
                             md_thermo* log, int64_t log_every) {
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state: call md_set_state or md_init_lattice first");
  if (!(dt > 0) || !std::isfinite(dt)) return fail(s, MD_ERR_INVALID_ARG, "dt must be > 0");
  if (nsteps < 0) return fail(s, MD_ERR_INVALID_ARG, "nsteps must be >= 0");
  if (log && log_every <= 0) return fail(s, MD_ERR_INVALID_ARG, "log_every must be > 0 when log is given");
  const int64_t nlog = (log && log_every > 0) ? nsteps / log_every : 0;
  CKS(ensure_thermo(s, nlog * s->nrep));
  // room for the partial records of up to MD_LOG_SLOTS NVE log steps per
  // launch (at most 256 MB), reduced after the launch's last step; the
  // Nose-Hoover kinds reduce every step anyway
  int slots = 0;
  if (nlog > 0 && kind != MD_KIND_NH && kind != MD_KIND_NH_EXACT && !s->log_now) {
    const size_t stride = (size_t)s->ntiles * list_lanes(s) * MD_NPART;
    const size_t most = ((size_t)256 << 20) / sizeof(double) / stride;
    slots = (int)std::min<int64_t>(std::min<int64_t>(nlog, MD_LOG_SLOTS), (int64_t)most);
    if (slots > 0 && (size_t)slots * stride > s->plog_cap) {
      dfree(s, s->d_plog);
      s->d_plog = nullptr;
      s->plog_cap = 0;
      CKS(dalloc(s, &s->d_plog, (size_t)slots * stride));
      s->plog_cap = (size_t)slots * stride;
    }
  }
  s->plog_slots = slots;
  int64_t done = 0;
  md_status st = run_op(s, MD_OP_STEPS, kind, dt, nsteps, nstep_boltz, seed, log ? log_every : 0, nlog, &done);
  s->plog_slots = 0;
  if (st != MD_OK) return st;
  if (nlog > 0) {
    CK(cudaMemcpyAsync(log, s->d_thermo, sizeof(ThermoDev) * nlog * s->nrep, cudaMemcpyDeviceToHost, s->stream));
    CK(cudaStreamSynchronize(s->stream));
  }
  return MD_OK;
}

md_status md_step_nve(md_system* s, double dt, int64_t nsteps, md_thermo* log, int64_t log_every) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  return step_common(s, MD_KIND_NVE, dt, nsteps, 0, 0, log, log_every);
}

md_status md_step_nvt(md_system* s, double dt, int64_t nsteps, const double* T_target, md_thermostat kind, double param,
                      uint64_t seed, md_thermo* log, int64_t log_every) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!T_target) return fail(s, MD_ERR_INVALID_ARG, "T_target must not be NULL");
  for (int r = 0; r < s->nrep; ++r)
    if (!(T_target[r] >= 0) || !std::isfinite(T_target[r])) return fail(s, MD_ERR_INVALID_ARG, "T_target must be >= 0");
  int k;
  int64_t nb = 0;
  if (kind == MD_NVT_NOSE_HOOVER || kind == MD_NVT_NOSE_HOOVER_EXACT) {
    if (!(param > 0)) return fail(s, MD_ERR_INVALID_ARG, "Nose-Hoover needs tau > 0");
    for (int r = 0; r < s->nrep; ++r)
      if (!(T_target[r] > 0)) return fail(s, MD_ERR_INVALID_ARG, "Nose-Hoover needs T_target > 0");
    k = kind == MD_NVT_NOSE_HOOVER ? MD_KIND_NH : MD_KIND_NH_EXACT;
  } else if (kind == MD_NVT_RESAMPLE) {
    nb = (int64_t)param;
    if (nb < 1) return fail(s, MD_ERR_INVALID_ARG, "resampling needs nstep_boltz >= 1");
    k = MD_KIND_RESAMPLE;
  } else {
    return fail(s, MD_ERR_INVALID_ARG, "unknown thermostat");
  }
  CKS(download_reps(s));
  for (int r = 0; r < s->nrep; ++r) {
    RepDev& R = s->reps[r];
    R.T_target = T_target[r];
    if (k != MD_KIND_RESAMPLE) R.Q = (double)s->ndim * R.n * T_target[r] * param * param;
  }
  s->reps_dirty = true;
  return step_common(s, k, dt, nsteps, nb, seed, log, log_every);
}

md_status md_rdf(md_system* s, double dr, int64_t nbins, double* g, int reset) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state");
  if (s->ntypes != 2) return fail(s, MD_ERR_INVALID_ARG, "md_rdf needs a 2-type system");
  if (!(dr > 0) || nbins < 1) return fail(s, MD_ERR_INVALID_ARG, "dr > 0 and nbins >= 1 required");
  for (int r = 0; r < s->nrep; ++r)
    if (dr * nbins > 0.5 * s->L_per[r] * (1 + 1e-12)) return fail(s, MD_ERR_INVALID_ARG, "nbins*dr must be <= L/2");
  if (reset || !s->d_rdf || nbins != s->rdf_nbins || dr != s->rdf_dr) {
    if (!s->d_rdf || nbins != s->rdf_nbins) {
      dfree(s, s->d_rdf);
      s->rdf_nbins = 0;
      CKS(dalloc(s, &s->d_rdf, (size_t)s->nrep * 3 * nbins));
    } else {
      CK(cudaMemsetAsync(s->d_rdf, 0, 8 * (size_t)s->nrep * 3 * nbins, s->stream));
    }
    s->rdf_nbins = nbins;
    s->rdf_dr = dr;
    s->rdf_meas = 0;
  }
  // the histogram walks the cell lists of the last build: make them current
  CKS(download_ctl(s));
  if (s->ctl.pending & MD_FLAG_REBUILD) CKS(run_op(s, MD_OP_REBUILD, MD_KIND_NVE, 0, 0, 0, 0, 0, 0, nullptr));
  CKS(download_ctl(s));
  RdfArgs a;
  a.mixed = s->mixed;
  a.ntot = s->ntot;
  a.nbins = (int)nbins;
  a.ndim = s->ndim;
  a.nrep = s->nrep;
  a.dr = dr;
  a.skin = s->tun.skin_outer;
  a.iunit = 1.0 / s->unit;
  a.reps = s->d_reps;
  a.tile_rep = s->d_tile_rep;
  a.xbq = s->d_xbq;
  // (two arrays of a rebuild, which has no use for them now: 32 entries per replica at least)
  a.unit = s->d_scat;
  a.nunits = s->d_cellof;
  a.nowhere = s->d_cellof + s->nrep;
  int32_t* const blk = s->d_cellof + 2 * (int64_t)s->nrep;
  a.blk = blk;
  a.pq = s->d_pq[s->ctl.cur];
  a.pfx = s->d_pfx;
  a.p4 = s->d_p4[s->ctl.cur];
  a.cstart = s->d_cstart;
  a.hist = s->d_rdf;
  // about eight CTAs per SM, shared out over the replicas by their candidate
  // pairs, at most one warp per unit (a unit holds 8 particles or more in
  // anything but a gas). With as many for each replica, one of 120 000 particles
  // among 1215 of two had one CTA: all pairs to L/2 6.4 s, now 27 ms.
  std::vector<double> work((size_t)s->nrep);
  double total = 0.0;
  for (int r = 0; r < s->nrep; ++r) {
    const RepDev& R = s->reps[r];
    int l;
    double share = 0.5;
    if (rdf_layers((dr * nbins + a.skin) * a.iunit, R.nc, R.cellw, &l))
      share = std::min(0.5, (2.0 * l + RDF_CELLS) * (l + 1.0) * (s->ndim == 3 ? 2.0 * l + 1.0 : 1.0) /
                                std::pow((double)R.nc, (double)s->ndim));
    work[r] = (double)R.n * (double)R.n * share;
    total += work[r];
  }
  s->rdf_blk.assign(1, 0);
  for (int r = 0; r < s->nrep; ++r) {
    const int64_t most = (s->n_per[r] / 8 + RDF_WARPS) / RDF_WARPS;
    const int64_t fair = (int64_t)std::ceil(8.0 * s->nsm * work[r] / total);
    s->rdf_blk.push_back(s->rdf_blk.back() + (int32_t)std::max<int64_t>(1, std::min(most, fair)));
  }
  CK(cudaMemsetAsync(a.nunits, 0, 8 * (size_t)s->nrep, s->stream));
  if (s->nrep > 1)
    CK(cudaMemcpyAsync(blk, s->rdf_blk.data(), 4 * s->rdf_blk.size(), cudaMemcpyHostToDevice, s->stream));
  k_rdf_units<<<blocks_for(s->ntot, RDF_LIST), RDF_LIST, 0, s->stream>>>(a);
  CK(cudaGetLastError());
  k_rdf<<<(unsigned)s->rdf_blk.back(), 32 * RDF_WARPS, 0, s->stream>>>(a);
  CK(cudaGetLastError());
  s->rdf_meas += 1;
  if (g) {
    std::vector<unsigned long long> h((size_t)s->nrep * 3 * nbins);
    CK(cudaMemcpyAsync(h.data(), s->d_rdf, 8 * h.size(), cudaMemcpyDeviceToHost, s->stream));
    CK(cudaStreamSynchronize(s->stream));
    for (int64_t k = 0; k < 3 * nbins; ++k) g[k] = 0.0;
    for (int r = 0; r < s->nrep; ++r) {
      const int64_t na = s->n_type0[r], nb = s->n_per[r] - na;
      // V and the shell volume of bin k; in two dimensions the area L^2 and the ring pi((k+1)^2 - k^2)dr^2
      const double Lr = s->L_per[r];
      const double V = s->ndim == 3 ? Lr * Lr * Lr : Lr * Lr;
      for (int64_t k = 0; k < nbins; ++k) {
        const double shell =
            s->ndim == 3 ? 4.0 / 3.0 * M_PI * (std::pow((double)(k + 1), 3) - std::pow((double)k, 3)) * dr * dr * dr
                         : M_PI * (std::pow((double)(k + 1), 2) - std::pow((double)k, 2)) * dr * dr;
        const unsigned long long* hr = h.data() + (size_t)r * 3 * nbins;
        const double m = (double)s->rdf_meas * s->nrep;
        if (na > 1) g[k] += hr[k] / shell * V / ((double)na * (na - 1)) / m;
        if (nb > 1) g[nbins + k] += hr[nbins + k] / shell * V / ((double)nb * (nb - 1)) / m;
        if (na > 0 && nb > 0) g[2 * nbins + k] += hr[2 * nbins + k] / shell * V / ((double)na * nb) / m;
      }
    }
  }
  return MD_OK;
}

md_status md_msd_tw(md_system* s, int slot, double* msd_per_type, int reset_reference) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state");
  if (slot < 0 || slot >= MD_MSD_SLOTS) return fail(s, MD_ERR_INVALID_ARG, "MSD slot out of range");
  CKS(download_ctl(s));
  if (reset_reference) CKS(reset_msd_ref(s, slot));
  if (!s->msd_valid[slot]) return fail(s, MD_ERR_INVALID_ARG, "MSD slot has no reference (reset it first)");
  const int nb = std::min(MSD_BLOCKS, (s->ntiles + MSD_THREADS / 32 - 1) / (MSD_THREADS / 32));
  k_msd_blocks<<<nb, MSD_THREADS, 0, s->stream>>>(s->mixed, s->ntypes, s->ntot, s->d_reps, s->d_tile_rep, s->d_pfx,
                                                  s->d_p4[s->ctl.cur], s->d_gid, s->d_typ, s->d_img,
                                                  s->d_msd_ref[slot], s->d_msd_part);
  CK(cudaGetLastError());
  k_msd_final<<<1, MSD_THREADS, 0, s->stream>>>(nb, s->ntypes, s->d_msd_part, s->d_io);
  CK(cudaGetLastError());
  if (msd_per_type) CK(cudaMemcpyAsync(msd_per_type, s->d_io, 8 * s->ntypes, cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  return MD_OK;
}

md_status md_msd(md_system* s, double* msd_per_type, int reset_reference) {
  return md_msd_tw(s, 0, msd_per_type, reset_reference);
}

md_status md_set_tuning(md_system* s, const md_tuning* t) {
  if (!s || !t) return fail(s, MD_ERR_INVALID_ARG, "NULL argument");
  CKS(tuning_ok(s, t));
  CKS(download_reps(s));
  s->tun = *t;
  layout_cells(s);
  for (auto& R : s->reps) R.want_rebuild = 1;
  s->stage_cap = stage_capacity(s);  // also picks each replica's group shape
  CKS(upload_reps(s));
  CKS(alloc_cells_and_list(s, list_capacity(s)));
  CKS(configure_grid(s));
  CKS(download_ctl(s));
  s->ctl.pending |= MD_FLAG_REBUILD;
  return MD_OK;
}

// fixed_skin > 0: the force list's skin stays fixed_skin and only the outer
// skin is searched; otherwise both are.
static md_status autotune_impl(md_system* s, double dt, int64_t probe_steps, double fixed_skin, md_tuning* best,
                               double* seconds_per_step) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state");
  if (!(dt > 0) || probe_steps < 1) return fail(s, MD_ERR_INVALID_ARG, "dt > 0 and probe_steps >= 1 required");
  // save the state (caller order, device) and the per-replica bath state
  const size_t n3 = 3 * (size_t)s->n_total;
  double* saved = nullptr;
  int32_t* saved_img = nullptr;
  CKS(dalloc(s, &saved, 2 * n3));
  CKS(dalloc(s, &saved_img, n3));
  md_status st = md_get_state(s, saved, saved + n3, saved_img, 1);
  if (st != MD_OK) { dfree(s, saved); dfree(s, saved_img); return st; }
  CKS(download_reps(s));
  const std::vector<RepDev> saved_reps = s->reps;
  const int64_t saved_step = s->ctl.step;
  const md_tuning start = s->tun;
  md_tuning bt = start;
  // starting skins of the first search stage
  const double s0 = fixed_skin > 0 ? fixed_skin : start.skin;
  const double so0 = fixed_skin > 0 ? fixed_skin : start.skin_outer;
  float bms = 1e30f;
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  // one probe: set the candidate, restart from the saved state, warm up,
  // then time probe_steps NVE steps
  auto probe = [&](const md_tuning& c) {
    if (st != MD_OK) return;
    if (c.block_size < 32 * c.threads_per_atom) return;
    // fewer lanes than the lists get: the same program as more (see list_lanes)
    if (!s->mixed && c.threads_per_atom < 4) return;
    if (tuning_ok(s, &c) != MD_OK) return;
    st = md_set_tuning(s, &c);
    if (st == MD_OK) st = set_state_impl(s, saved, saved + n3, 1);
    if (st == MD_OK) st = md_step_nve(s, dt, std::max<int64_t>(probe_steps / 4, 1), nullptr, 0);
    if (st != MD_OK) return;
    cudaEventRecord(e0, s->stream);
    st = md_step_nve(s, dt, probe_steps, nullptr, 0);
    cudaEventRecord(e1, s->stream);
    cudaEventSynchronize(e1);
    float ms = 0;
    cudaEventElapsedTime(&ms, e0, e1);
    if (st == MD_OK && ms < bms) { bms = ms; bt = c; }
  };
  const int Ts[4] = {1, 2, 4, 8};
  const int Bs[3] = {128, 256, 512};
  // (skin, skin_outer); equal values mean one list without pruning
  const double Sfree[9][2] = {{0.2, 0.2}, {0.3, 0.3}, {0.4, 0.4}, {0.2, 0.5}, {0.2, 0.7},
                              {0.3, 0.6}, {0.3, 0.8}, {0.3, 1.0}, {0.4, 0.9}};
  double Ss[9][2];
  int nS = 0;
  if (fixed_skin > 0) {
    const double extra[6] = {0.0, 0.3, 0.5, 0.7, 0.9, 1.1};
    for (int k = 0; k < 6; ++k) { Ss[nS][0] = fixed_skin; Ss[nS][1] = fixed_skin + extra[k]; ++nS; }
  } else {
    for (int k = 0; k < 9; ++k) { Ss[nS][0] = Sfree[k][0]; Ss[nS][1] = Sfree[k][1]; ++nS; }
  }
  // coordinate search: lanes x block size at the starting skins, then the
  // skins at the best of those, then lanes x block size again at the best skins
  for (int ti = 0; ti < 4; ++ti)
    for (int bi = 0; bi < 3; ++bi) probe(md_tuning{Ts[ti], Bs[bi], s0, so0});
  const md_tuning b1 = bt;
  for (int si = 0; si < nS; ++si)
    if (!(Ss[si][0] == s0 && Ss[si][1] == so0))
      probe(md_tuning{b1.threads_per_atom, b1.block_size, Ss[si][0], Ss[si][1]});
  const md_tuning b2 = bt;
  if (!(b2.skin == s0 && b2.skin_outer == so0))
    for (int ti = 0; ti < 4; ++ti)
      for (int bi = 0; bi < 3; ++bi)
        if (!(Ts[ti] == b2.threads_per_atom && Bs[bi] == b2.block_size))
          probe(md_tuning{Ts[ti], Bs[bi], b2.skin, b2.skin_outer});
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  md_status st2 = md_set_tuning(s, st == MD_OK ? &bt : &start);
  if (st2 == MD_OK) st2 = set_state_impl(s, saved, saved + n3, 1);
  if (st2 == MD_OK) {
    const int b = 256;
    k_set_images<<<blocks_for(s->n_total, b), b, 0, s->stream>>>(s->n_total, s->ntot, s->d_reps, s->d_rep_of_caller,
                                                                 saved_img, s->d_img);
    cudaError_t ce = cudaGetLastError();
    if (ce != cudaSuccess) st2 = cuda_fail(s, ce, "k_set_images");
  }
  if (st2 == MD_OK) st2 = download_reps(s);
  if (st2 == MD_OK) {
    for (int r = 0; r < s->nrep; ++r) {
      RepDev& R = s->reps[r];
      const RepDev& O = saved_reps[r];
      R.T_target = O.T_target; R.Q = O.Q; R.xi = O.xi; R.g = O.g; R.lns = O.lns; R.lns_next = O.lns_next;
      R.xi_a = O.xi_a; R.rebuilds = O.rebuilds;
    }
    s->reps_dirty = true;
    s->ctl.step = saved_step;
  }
  if (st2 == MD_OK) st2 = reset_msd_ref(s);
  cudaStreamSynchronize(s->stream);
  dfree(s, saved);
  dfree(s, saved_img);
  if (st != MD_OK) return st;
  if (st2 != MD_OK) return st2;
  if (best) *best = bt;
  if (seconds_per_step) *seconds_per_step = (double)bms * 1e-3 / (double)probe_steps;
  return MD_OK;
}

md_status md_autotune(md_system* s, double dt, int64_t probe_steps, md_tuning* best, double* seconds_per_step) {
  return autotune_impl(s, dt, probe_steps, -1.0, best, seconds_per_step);
}

md_status md_autotune_skin(md_system* s, double dt, int64_t probe_steps, double skin, md_tuning* best,
                           double* seconds_per_step) {
  if (!(skin >= 0.05) || !(skin < 2.0)) return fail(s, MD_ERR_INVALID_ARG, "skin must be in [0.05, 2)");
  return autotune_impl(s, dt, probe_steps, skin, best, seconds_per_step);
}

md_status md_time_forces(md_system* s, int64_t repeats, double* seconds_per_eval) {
  if (!s || !seconds_per_eval) return fail(s, MD_ERR_INVALID_ARG, "NULL argument");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state: call md_set_state or md_init_lattice first");
  if (repeats < 1 || repeats > 100000) return fail(s, MD_ERR_INVALID_ARG, "repeats must be in [1, 100000]");
  // bring the lists up to date first (a rebuild would otherwise be timed too)
  CKS(download_ctl(s));
  if (s->ctl.drifted) return fail(s, MD_ERR_INVALID_ARG, "the state is between a position and a velocity update");
  if (s->ctl.pending & (MD_FLAG_REBUILD | MD_FLAG_PRUNE))
    CKS(run_op(s, MD_OP_REBUILD, MD_KIND_NVE, 0, 0, 0, 0, 0, 0, nullptr));
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  md_status st = MD_OK;
  float ms = 0.0f, ms1 = 0.0f;
  // the launch's fixed cost (start, first barrier, end) is taken out by a
  // launch with one evaluation: seconds = (t(repeats) - t(1)) / (repeats - 1)
  for (int pass = 0; pass < 2 && st == MD_OK; ++pass) {
    const int64_t k = pass == 0 ? 1 : repeats;
    cudaEventRecord(e0, s->stream);
    st = run_op(s, MD_OP_FORCE_REPEAT, MD_KIND_NVE, 0.0, k, 0, 0, 0, 0, nullptr);
    cudaEventRecord(e1, s->stream);
    cudaEventSynchronize(e1);
    cudaEventElapsedTime(pass == 0 ? &ms1 : &ms, e0, e1);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != MD_OK) return st;
  *seconds_per_eval = repeats > 1 ? (double)(ms - ms1) * 1e-3 / (double)(repeats - 1) : (double)ms * 1e-3;
  return MD_OK;
}

md_status md_time_lists(md_system* s, int64_t repeats, double* seconds_per_build) {
  if (!s || !seconds_per_build) return fail(s, MD_ERR_INVALID_ARG, "NULL argument");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state: call md_set_state or md_init_lattice first");
  if (repeats < 2 || repeats > 10000) return fail(s, MD_ERR_INVALID_ARG, "repeats must be in [2, 10000]");
  CKS(download_ctl(s));
  if (s->ctl.drifted) return fail(s, MD_ERR_INVALID_ARG, "the state is between a position and a velocity update");
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  md_status st = MD_OK;
  float ms = 0.0f, ms1 = 0.0f;
  // both launches start with the same full rebuild, which the difference
  // takes out with the launch's fixed cost
  for (int pass = 0; pass < 2 && st == MD_OK; ++pass) {
    const int64_t k = pass == 0 ? 1 : repeats;
    st = mark_rebuild_all(s);
    if (st != MD_OK) break;
    cudaEventRecord(e0, s->stream);
    st = run_op(s, MD_OP_LIST_REPEAT, MD_KIND_NVE, 0.0, k, 0, 0, 0, 0, nullptr);
    cudaEventRecord(e1, s->stream);
    cudaEventSynchronize(e1);
    cudaEventElapsedTime(pass == 0 ? &ms1 : &ms, e0, e1);
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st != MD_OK) return st;
  *seconds_per_build = (double)(ms - ms1) * 1e-3 / (double)(repeats - 1);
  return MD_OK;
}

md_status md_get_tuning(const md_system* s, md_tuning* t) {
  if (!s || !t) return MD_ERR_INVALID_ARG;
  *t = s->tun;
  return MD_OK;
}

md_status md_get_info(md_system* s, md_info* info) {
  if (!s || !info) return fail(s, MD_ERR_INVALID_ARG, "NULL argument");
  CKS(download_reps(s));
  CKS(download_ctl(s));
  std::memset(info, 0, sizeof(*info));
  info->n_total = s->n_total;
  info->n_replicas = s->nrep;
  info->grid_blocks = s->shape[0].grid;
  info->steps_done = s->ctl.step;
  for (const auto& R : s->reps) {
    info->rebuilds += R.rebuilds;
    info->all_pairs_replicas += R.nc == 0;
  }
  CK(cudaMemsetAsync(s->d_count, 0, 8, s->stream));
  // entries of the list the force phase reads: the inner list when there are two
  const bool dual = s->tun.skin_outer > s->tun.skin;
  k_sum_i32<<<std::max(1, std::min(1024, blocks_for(s->ntot * list_lanes(s), 256))), 256, 0, s->stream>>>(
      s->ntot * list_lanes(s), dual ? s->d_nnb_in : s->d_nnb, s->d_count);
  CK(cudaGetLastError());
  unsigned long long entries = 0;
  CK(cudaMemcpyAsync(&entries, s->d_count, 8, cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  info->list_entries = (int64_t)entries;
  info->list_capacity = (int64_t)s->maxrows * list_lanes(s);
  info->device_bytes = (int64_t)s->bytes;
  info->precision = s->mixed ? MD_PREC_MIXED : MD_PREC_FP64;
  info->graph_launches = s->graph_launches;
  info->prunes = s->ctl.prunes;
  info->kernel_launches = s->kernel_launches;
  return MD_OK;
}

md_status md_count_pairs(md_system* s, int64_t* pairs) {
  if (!s || !pairs) return fail(s, MD_ERR_INVALID_ARG, "NULL argument");
  if (!s->have_state) return fail(s, MD_ERR_INVALID_ARG, "no state");
  CKS(download_ctl(s));
  if (s->ctl.pending & MD_FLAG_REBUILD) CKS(run_op(s, MD_OP_REBUILD, MD_KIND_NVE, 0, 0, 0, 0, 0, 0, nullptr));
  CKS(download_ctl(s));
  double rc2d[16];
  for (int t = 0; t < s->ntypes * s->ntypes; ++t) rc2d[t] = s->rc[t] * s->rc[t];
  CK(cudaMemcpyAsync(s->d_io, rc2d, sizeof(double) * s->ntypes * s->ntypes, cudaMemcpyHostToDevice, s->stream));
  CK(cudaMemsetAsync(s->d_count, 0, 8, s->stream));
  const int b = 128;
  k_count_pairs<<<blocks_for(s->ntot, b), b, 0, s->stream>>>(
      s->mixed, s->ntot, s->ntypes, (rc_max(s) + s->tun.skin_outer) / s->unit, s->d_reps, s->d_tile_rep, s->d_pfx,
      s->d_p4[s->ctl.cur], s->d_typ, s->d_cstart, s->d_io, s->d_count);
  CK(cudaGetLastError());
  unsigned long long c = 0;
  CK(cudaMemcpyAsync(&c, s->d_count, 8, cudaMemcpyDeviceToHost, s->stream));
  CK(cudaStreamSynchronize(s->stream));
  *pairs = (int64_t)c;
  return MD_OK;
}

md_status md_selftest_barrier(md_system* s, double timeout_s) {
  if (!s) return fail(nullptr, MD_ERR_INVALID_ARG, "NULL system");
  if (!(timeout_s > 0) || timeout_s > 60) return fail(s, MD_ERR_INVALID_ARG, "timeout_s must be in (0, 60]");
  CKS(download_ctl(s));
  const CtlDev saved = s->ctl;
  s->ctl.pending = 0;
  CKS(upload_state(s));
  KParams p = make_params(s);
  p.timeout_ns = (unsigned long long)(timeout_s * 1e9);
  s->ctl_now = false;
  CK(md_launch_barrier_selftest(p, 4, s->stream));
  CKS(download_ctl(s));
  const int pend = s->ctl.pending;
  // restore the control block so the system stays usable
  s->ctl = saved;
  if (pend & MD_FLAG_TIMEOUT) return fail(s, MD_ERR_TIMEOUT, "barrier wait ran out as intended (self-test)");
  return fail(s, MD_ERR_CUDA, "barrier self-test: the wait did not run out");
}

#ifdef KAMD_PHASE_TIMERS
// profiling builds only: copy out (and clear) the per-barrier phase timers
md_status md_debug_phase_times(md_system* s, double* ns, double* cnt) {
  CKS(download_ctl(s));
  for (int k = 0; k < 128; ++k) {
    ns[k] = (double)s->ctl.phase_ns[k];
    cnt[k] = (double)s->ctl.phase_cnt[k];
    s->ctl.phase_ns[k] = 0;
    s->ctl.phase_cnt[k] = 0;
  }
  s->ctl.t_last = 0;
  return MD_OK;
}
#endif

const char* md_last_error(const md_system* s) {
  if (!s) return g_create_err.c_str();
  return s->err.c_str();
}

void md_destroy(md_system* s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  for (auto& h : s->shape) drop_graph(h);
  if (s->h_land) cudaFreeHost(s->h_land);
  dfree(s, s->d_state); dfree(s, s->d_tile_rep);
  dfree(s, s->d_pfx); dfree(s, s->d_pq[0]); dfree(s, s->d_pq[1]); dfree(s, s->d_velf); dfree(s, s->d_frcf); dfree(s, s->d_xbq);
  dfree(s, s->d_xbq_in); dfree(s, s->d_nbr_in); dfree(s, s->d_nnb_in);
  dfree(s, s->d_p4[0]); dfree(s, s->d_p4[1]); dfree(s, s->d_veld); dfree(s, s->d_frcd);
  dfree(s, s->d_gid); dfree(s, s->d_typ); dfree(s, s->d_img);
  dfree(s, s->d_tpfx); dfree(s, s->d_tp4); dfree(s, s->d_tvel); dfree(s, s->d_tfrc); dfree(s, s->d_tgid); dfree(s, s->d_ttyp);
  dfree(s, s->d_timg);
  dfree(s, s->d_cellof); dfree(s, s->d_cell_rep); dfree(s, s->d_ccount); dfree(s, s->d_cstart); dfree(s, s->d_ccursor); dfree(s, s->d_chunk); dfree(s, s->d_cta_sm); dfree(s, s->d_redmap); dfree(s, s->d_redrep); dfree(s, s->d_redpart); dfree(s, s->d_scat);
  dfree(s, s->d_nbr); dfree(s, s->d_nnb); dfree(s, s->d_part[0]); dfree(s, s->d_part[1]); dfree(s, s->d_plog); dfree(s, s->d_plog_rec);
  dfree(s, s->d_typ_caller); dfree(s, s->d_rep_of_caller); dfree(s, s->d_thermo); dfree(s, s->d_io);
  dfree(s, s->d_io_i); dfree(s, s->d_rdf); dfree(s, s->d_msd_part); dfree(s, s->d_count);
  for (int k = 0; k < MD_MSD_SLOTS; ++k) dfree(s, s->d_msd_ref[k]);
  delete s;
}

}  // extern "C"
