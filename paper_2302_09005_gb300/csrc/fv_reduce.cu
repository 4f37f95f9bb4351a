// fv_reduce.cu -- maximum eigenvalue per patch and over the batch with the
// CFL time step (Eq. 5, Algorithm 1 step 10), and the fixed-order FP64
// conservation sums.
#include "fv_device.cuh"
#include "fv_internal.h"
#include "fv_ptx.cuh"

namespace fv {

// ---------------------------------------------------------------------------
// Maximum eigenvalue.  The per-patch value is the largest a over the faces
// that bound interior cells; a face's a is the larger |u_k| + c of its two
// cells, so the patch value is the maximum of |u_k| + c over the interior
// cells (every k) and the face-halo cells (their normal k only).  One warp per
// patch (four per CTA, grid stride over the warps), the patch maximum by warp
// shuffles; cells are read straight from HBM, as 16-byte words where a cell's
// size is a multiple of 16 bytes (2D).
// ---------------------------------------------------------------------------
template <typename T>
struct EigParams {
  const T* q;
  const int64_t* off;
  const int32_t* sizes;
  int64_t n;
  int halo;
  int pmax;
  T gamma, gm1;
  double* per_patch;
  unsigned long long* partials;
  unsigned int* status;
};

template <int D>
__device__ __forceinline__ int64_t ipow64(int b) {
  return D == 1 ? b : D == 2 ? (int64_t)b * b : (int64_t)b * b * b;
}

// Element offset of cell t of a patch (its interior cells, then the face-halo
// cells of its 2D faces); kdir: the direction whose wave speed counts (-1: all).
template <int D>
__device__ __forceinline__ int eig_cell(int t, int p, int h, int ne, int nint, int ptr,
                                        int& kdir) {
  int c[3] = {0, 0, 0};
  kdir = -1;
  if (t < nint) {
    int r = t;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      c[k] = h + r % p;
      r /= p;
    }
  } else {
    const int j = t - nint;
    const int f = j / ptr;
    int r = j - f * ptr;
    kdir = f >> 1;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      if (k != kdir) {
        c[k] = h + r % p;
        r /= p;
      } else {
        c[k] = (f & 1) ? h + p : h - 1;
      }
    }
  }
  int cid = c[D - 1];
#pragma unroll
  for (int k = D - 2; k >= 0; --k) cid = cid * ne + c[k];
  return cid * (D + 2);
}
template <typename T, int S>
__device__ __forceinline__ void eig_load(const T* src, T (&q)[S]) {
  if constexpr ((S * sizeof(T)) % 16 == 0) {
#pragma unroll
    for (int u = 0; u < (int)(S * sizeof(T) / 16); ++u) {
      const uint4 w = reinterpret_cast<const uint4*>(src)[u];
      memcpy(&q[u * (16 / sizeof(T))], &w, 16);
    }
  } else {
#pragma unroll
    for (int v = 0; v < S; ++v) q[v] = src[v];
  }
}
// The largest |u_k| + c of a cell (over every k, or kdir alone), as bits.
template <typename T, int D>
__device__ __forceinline__ unsigned long long eig_value(const T* q, T gm1, T gamma, int kdir,
                                                        bool& bad) {
  const Prim<T, D> w = primitives<T, D>(q, gm1, gamma, bad);
  unsigned long long m = 0ull;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    if (kdir < 0 || kdir == k) {
      const unsigned long long b = order_bits(add_rn(abs_t(w.u[k]), w.c));
      m = b > m ? b : m;
    }
  }
  return m;
}

// FP64: FP32 bounds of every cell first (wave_bounds), then the FP64 wave
// speed of the cells whose upper bound reaches the patch's largest lower bound
// (or, where only the batch maximum is asked for, the warp's largest wave
// speed so far).  Where the states vary from cell to cell that is one cell or
// two of a patch, and the kernel leaves the FP64 pipe, which bound it when every
// cell was converted in FP64 (random states, 262,144 patches of 5^3: 3.08 ms,
// now 0.82 with the per-patch values and 0.72 without; 40,000 of 7^3: 1.07 ->
// 0.25).  Where the wave speed is constant over a patch every cell is a
// candidate and is loaded again for FP64: 32,768 patches of 5^3 395 -> 235 us for
// a uniform moving state, 395 -> 333 for a blast into gas at rest, 108 for random
// states.  The maximum is exact all the same.
template <typename T, int D>
__global__ void __launch_bounds__(FV_NT) eig_kernel(EigParams<T> a) {
  constexpr int S = D + 2;
  constexpr int VEC = 16 / sizeof(T);
  constexpr int NW = FV_NT / 32;
  __shared__ unsigned long long red[NW];
  grid_dep_wait();
  grid_dep_launch();
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t step = (int64_t)gridDim.x * NW;
  unsigned long long warp_max = 0ull;  // over this warp's patches
  int64_t i = (int64_t)blockIdx.x * NW + (tid >> 5);
  int pn = 0;  // the next patch's metadata, loaded one patch ahead
  int64_t offn = 0;
  if (i < a.n) {
    pn = a.sizes[i];
    offn = a.off[i];
  }
  for (; i < a.n; i += step) {
    const int p = pn;
    const int64_t off = offn;
    if (i + step < a.n) {
      pn = a.sizes[i + step];
      offn = a.off[i + step];
    }
    const int h = a.halo;
    if (!(p >= 1 && p <= a.pmax && off >= 0 && (off % VEC) == 0)) {
      if (lane == 0) atomicOr(a.status, ST_BAD_PATCH);
      continue;
    }
    const int ne = p + 2 * h;
    const int ptr = D == 1 ? 1 : D == 2 ? p : p * p;
    const int nint = ptr * p, ncell = nint + 2 * D * ptr;
    const T* Q = a.q + off;
    unsigned long long m = 0ull;
    bool bad = false;
    if (sizeof(T) == 4 || ncell <= 32) {  // a lane's one cell needs no sorting out
      for (int t = lane; t < ncell; t += 32) {
        int kdir;
        T q[S];
        eig_load<T, S>(Q + eig_cell<D>(t, p, h, ne, nint, ptr, kdir), q);
        const unsigned long long b = eig_value<T, D>(q, a.gm1, a.gamma, kdir, bad);
        m = b > m ? b : m;
      }
    } else if constexpr (sizeof(T) == 8) {
      const float gm1 = (float)a.gm1, gam = (float)a.gamma;
      // this lane's largest lower bound, its two largest upper bounds and the
      // cell of the largest
      float lo = 0.f, hi1 = -1.f, hi2 = -1.f;
      int best = lane;
      for (int t = lane; t < ncell; t += 32) {
        int kdir;
        T q[S];
        eig_load<T, S>(Q + eig_cell<D>(t, p, h, ne, nint, ptr, kdir), q);
        float l, u;
        wave_bounds<D>(q, gm1, gam, kdir, l, u);
        lo = fmaxf(lo, l);
        const bool top = u > hi1;
        hi2 = fmaxf(hi2, top ? hi1 : u);
        best = top ? t : best;
        hi1 = top ? u : hi1;
      }
      // lower bounds are >= 0, so their bits order like the values
      float thr = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(lo)));
      if (a.per_patch == nullptr) thr = fmaxf(thr, wave_floor(warp_max));
      if (hi1 >= thr) {
        const bool all = hi2 >= thr;
        for (int t = all ? lane : best; t < ncell; t += all ? 32 : ncell) {
          int kdir;
          T q[S];
          eig_load<T, S>(Q + eig_cell<D>(t, p, h, ne, nint, ptr, kdir), q);
          float l, u;
          wave_bounds<D>(q, gm1, gam, kdir, l, u);
          if (u >= thr) {
            const unsigned long long b = eig_value<T, D>(q, a.gm1, a.gamma, kdir, bad);
            m = b > m ? b : m;
          }
        }
      }
    }
    if (bad) atomicOr(a.status, ST_NONPHYSICAL);
    m = warp_max_u64(m);  // in every lane
    if (lane == 0 && a.per_patch) a.per_patch[i] = order_value<T>(m);
    warp_max = m > warp_max ? m : warp_max;
  }
  if (lane == 0) red[tid >> 5] = warp_max;
  __syncthreads();
  if (tid == 0) {
    unsigned long long mm = red[0];
#pragma unroll
    for (int w2 = 1; w2 < NW; ++w2) mm = red[w2] > mm ? red[w2] : mm;
    a.partials[blockIdx.x] = mm;
  }
}

// Reduces the per-CTA maxima (bit patterns of type T), writes the global
// maximum and dt = cfl dx / (d lambda_max).
struct EigFinish {
  const unsigned long long* partials;
  int nparts;
  double* global_out;
  unsigned long long* lam_slot;
  double* dt_slot;
  double* dt_out;
  double cfl, dx;
};
template <typename T, int D>
__global__ void eig_finish_kernel(EigFinish a) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ unsigned long long red[32];
  unsigned long long m = 0ull;
  for (int j = threadIdx.x; j < a.nparts; j += blockDim.x)
    m = a.partials[j] > m ? a.partials[j] : m;
  m = warp_max_u64(m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = red[w] > m ? red[w] : m;
    m = red[0] > m ? red[0] : m;
    const double lam = order_value<T>(m);
    if (a.global_out) *a.global_out = lam;
    *a.lam_slot = m;  // bits, read by the next time step
    const double dt = (a.cfl * a.dx) / ((double)D * lam);
    *a.dt_slot = dt;
    if (a.dt_out) *a.dt_out = dt;
  }
}

template <typename T, int D>
static cudaError_t launch_eig_t(const fv_batch* h, const EigLaunch& l, int grid) {
  EigParams<T> a;
  a.q = static_cast<const T*>(l.q);
  a.off = l.off;
  a.sizes = l.sizes;
  a.n = l.n;
  a.halo = l.halo;
  a.pmax = h->max_patch_size;
  a.gamma = (T)l.gamma;
  a.gm1 = (T)(l.gamma - 1.0);
  a.per_patch = l.per_patch;
  a.partials = l.partials;
  a.status = l.status;
  return launch_kernel(eig_kernel<T, D>, grid, FV_NT, 0, h->stream, starts_early(h, grid, FV_NT), a);
}

cudaError_t launch_eig(const fv_batch* h, const EigLaunch& l, int grid) {
  if (h->prec == FV_FP64) {
    if (h->d == 1) return launch_eig_t<double, 1>(h, l, grid);
    if (h->d == 2) return launch_eig_t<double, 2>(h, l, grid);
    return launch_eig_t<double, 3>(h, l, grid);
  }
  if (h->d == 1) return launch_eig_t<float, 1>(h, l, grid);
  if (h->d == 2) return launch_eig_t<float, 2>(h, l, grid);
  return launch_eig_t<float, 3>(h, l, grid);
}

cudaError_t launch_eig_finish(const fv_batch* h, const unsigned long long* partials, int nparts,
                              double* global_out, unsigned long long* lam_slot, double* dt_slot,
                              double* dt_out, double cfl, double dx) {
  const EigFinish a{partials, nparts, global_out, lam_slot, dt_slot, dt_out, cfl, dx};
#define FV_EIG_FIN(T, D) launch_kernel(eig_finish_kernel<T, D>, 1, 256, 0, h->stream, true, a)
  if (h->prec == FV_FP64)
    return h->d == 1   ? FV_EIG_FIN(double, 1)
           : h->d == 2 ? FV_EIG_FIN(double, 2)
                       : FV_EIG_FIN(double, 3);
  return h->d == 1   ? FV_EIG_FIN(float, 1)
         : h->d == 2 ? FV_EIG_FIN(float, 2)
                     : FV_EIG_FIN(float, 3);
#undef FV_EIG_FIN
}

// ---------------------------------------------------------------------------
// Conservation sums in FP64, fixed order: chunk c holds patches
// [c*FV_SUM_CHUNK, (c+1)*FV_SUM_CHUNK), cut into 128 slices: slice v adds
// patches v, v + 128, ... of the chunk in index order, each patch by a fixed
// cell-to-lane map and a fixed tree.  A cluster of eight CTAs sums a chunk, a
// warp a slice (or four, one after the other); the slices' sums meet in the
// first CTA's shared memory and are added by a fixed tree.  A final single CTA
// adds the chunks with a fixed tree.  The result does not depend on the CTA
// size, on the grid size or on timing.
//
// Bound by the latency of a warp's patch (its loads, then a tree of FP64 adds)
// where there are few chunks, which therefore take sixteen warps a CTA; with
// many, four warps a CTA at their higher occupancy are as good or better.
// Before, a CTA summed a chunk, all threads on one patch at a time (nine
// barriers a patch).  Before / sixteen / four warps, us: 9,177 patches of 6^3
// (FP64) 4050 / 95 / 187; 5,000 of 8^3 (FP32) 5537 / 134 / 328; 262,144 of
// 5^3 (FP64) 3601 / 1062 / 829; 670,761 of 5x5 (FP32) 3338 / 933 / 516.
// ---------------------------------------------------------------------------
template <typename T>
struct SumParams {
  const T* q;
  const int64_t* off;
  const int32_t* sizes;
  int64_t n;
  int halo;
  int pmax;
  double* partials;
  unsigned int* status;
  double* per_patch;
};

template <int S>
__device__ __forceinline__ void block_sum_fixed(double (&v)[S], double* sh /*[FV_NT][S]*/) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int k = 0; k < S; ++k) sh[tid * S + k] = v[k];
  __syncthreads();
  for (int w = FV_NT / 2; w > 0; w >>= 1) {
    if (tid < w) {
#pragma unroll
      for (int k = 0; k < S; ++k) sh[tid * S + k] = sh[tid * S + k] + sh[(tid + w) * S + k];
    }
    __syncthreads();
  }
#pragma unroll
  for (int k = 0; k < S; ++k) v[k] = sh[k];
  __syncthreads();
}

// A lane's S values summed over the warp (pairs at distance 16, 8, 4, 2, 1,
// in that order), with the lanes shared out: after the first steps half the
// lanes carry one unknown and half another, so the 5 S adds of S separate
// trees take 8 (S = 5).  Returns the sum of unknown sum_comp<S>(lane).
template <int S>
__device__ __forceinline__ int sum_comp(int lane) {
  const int b4 = (lane >> 4) & 1, b3 = (lane >> 3) & 1, b2 = (lane >> 2) & 1;
  if (S == 3) return b3 ? 2 : b4;
  return (S == 5 && b2) ? 4 : 2 * b3 + b4;
}
// Whether this lane is the one that stores its unknown's sum.
template <int S>
__device__ __forceinline__ bool sum_lane(int lane) {
  if ((lane & 3) != 0) return false;
  if (S == 5) return (lane & 4) == 0 || lane == 4;
  return (lane & 4) == 0 && !(S == 3 && lane == 24);
}
__device__ __forceinline__ double fold(double a, double b, int lane, int w) {
  const bool up = (lane & w) != 0;  // lower half keeps a, upper half b
  const double send = up ? a : b, keep = up ? b : a;
  return keep + __shfl_xor_sync(0xFFFFFFFFu, send, w);
}
__device__ __forceinline__ double fold1(double a, int w) {
  return a + __shfl_xor_sync(0xFFFFFFFFu, a, w);
}
template <int S>
__device__ __forceinline__ double warp_sums(const double (&v)[S], int lane) {
  const double r0 = fold(v[0], v[1], lane, 16);
  double t;
  if constexpr (S == 3) {
    t = fold(r0, fold1(v[2], 16), lane, 8);
    t = fold1(t, 4);
  } else {
    const double r1 = fold(v[2], v[3], lane, 16);
    t = fold(r0, r1, lane, 8);
    if constexpr (S == 5)
      t = fold(t, fold1(fold1(v[4], 16), 8), lane, 4);
    else
      t = fold1(t, 4);
  }
  return fold1(fold1(t, 2), 1);
}

// A float as a double: on the integer pipe but for subnormals (widen_f32
// flushes those).
__device__ __forceinline__ double widen(double x) { return x; }
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x) & 0x7FFFFFFFu;
  return u != 0u && u < 0x00800000u ? (double)x : widen_f32(x);
}

// The sums of one patch's interior, each unknown in the lanes of sum_comp;
// false: bad metadata.
template <typename T, int D>
__device__ __forceinline__ bool patch_sum(const SumParams<T>& a, int p, int64_t off, int lane,
                                          double& ps) {
  constexpr int S = D + 2;
  constexpr int VEC = 16 / sizeof(T);
  if (!(p >= 1 && p <= a.pmax && off >= 0 && (off % VEC) == 0)) return false;
  const int h = a.halo, ne = p + 2 * h;
  const int nint = D == 1 ? p : D == 2 ? p * p : p * p * p;
  // four accumulators a lane (cells lane + 32 m mod 128): independent loads
  double acc[4][S];
#pragma unroll
  for (int m = 0; m < 4; ++m)
#pragma unroll
    for (int k = 0; k < S; ++k) acc[m][k] = 0.0;
  for (int t0 = lane; t0 < nint; t0 += 128) {
    T v[4][S];
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int t = t0 + 32 * m;
#pragma unroll
      for (int k = 0; k < S; ++k) v[m][k] = T(0);
      if (t < nint) {
        int c[3] = {0, 0, 0};
        int r = t;
#pragma unroll
        for (int k = 0; k < D; ++k) {
          c[k] = h + r % p;
          r /= p;
        }
        int64_t cid = c[D - 1];
#pragma unroll
        for (int k = D - 2; k >= 0; --k) cid = cid * ne + c[k];
        const T* qc = a.q + off + cid * S;
#pragma unroll
        for (int k = 0; k < S; ++k) v[m][k] = qc[k];
      }
    }
    const bool head = t0 < 128;  // the first round starts the sums
#pragma unroll
    for (int m = 0; m < 4; ++m)
#pragma unroll
      for (int k = 0; k < S; ++k)
        acc[m][k] = head ? widen(v[m][k]) : acc[m][k] + widen(v[m][k]);
  }
  double s[S];
#pragma unroll
  for (int k = 0; k < S; ++k) {
    s[k] = acc[0][k];
    if (nint > 32) {
      if (nint > 64) s[k] = s[k] + acc[2][k];
      s[k] = s[k] + (nint > 96 ? acc[1][k] + acc[3][k] : acc[1][k]);
    }
  }
  ps = warp_sums<S>(s, lane);
  return true;
}

constexpr int kSumCluster = 8;   // CTAs per chunk
constexpr int kSumSlices = 128;  // per chunk
constexpr int kSumFewChunks = 32;  // up to here sixteen warps a CTA

template <typename T, int D, int NT>
__global__ void __cluster_dims__(kSumCluster, 1, 1) __launch_bounds__(NT)
    sums_kernel(SumParams<T> a) {
  constexpr int S = D + 2;
  constexpr int NW = kSumCluster * (NT / 32);  // warps per chunk
  static_assert(kSumSlices % NW == 0, "every warp takes as many slices");
  __shared__ double sh[kSumSlices * S];  // used in the cluster's first CTA
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  const int lane = threadIdx.x & 31;
  const int rank = blockIdx.x % kSumCluster;
  const int64_t chunk = blockIdx.x / kSumCluster;
  int v = rank * (NT / 32) + (threadIdx.x >> 5);  // the warp's slice
  const int64_t i0 = chunk * FV_SUM_CHUNK;
  const int64_t i1 = i0 + FV_SUM_CHUNK < a.n ? i0 + FV_SUM_CHUNK : a.n;
  const int comp = sum_comp<S>(lane);
  uint32_t dst;
  {
    const uint32_t own = smem_addr(sh);
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(own), "r"(0));
  }
  // the first CTA's shared memory may be written once every CTA has started
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  double total = 0.0;  // of unknown comp over the slice so far
  grid_dep_wait();
  grid_dep_launch();
  int64_t i = i0 + v;
  int pn = 0;  // the next patch's metadata, loaded one patch ahead
  int64_t offn = 0;
  if (i < i1) {
    pn = a.sizes[i];
    offn = a.off[i];
  }
  for (; v < kSumSlices;) {
    const int64_t cur = i;
    const bool on = cur < i1;  // else: a slice without patches
    const int p = pn;
    const int64_t off = offn;
    i += kSumSlices;
    const bool last = i >= i1;  // of the slice
    const int sl = v;
    if (last) {
      v += NW;
      i = i0 + v;
    }
    if (v < kSumSlices && i < i1) {
      pn = a.sizes[i];
      offn = a.off[i];
    }
    if (on) {
      double ps;
      if (patch_sum<T, D>(a, p, off, lane, ps)) {
        if (a.per_patch != nullptr && sum_lane<S>(lane)) a.per_patch[cur * S + comp] = ps;
        total = total + ps;
      } else if (lane == 0) {
        atomicOr(a.status, ST_BAD_PATCH);
      }
    }
    if (last) {  // the slice's sum to the cluster's first CTA
      if (sum_lane<S>(lane))
        asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(dst + 8u * (sl * S + comp)),
                     "d"(total)
                     : "memory");
      total = 0.0;
    }
  }
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
  if (rank == 0 && threadIdx.x < 32) {
    double t4[S];
#pragma unroll
    for (int k = 0; k < S; ++k) {
      t4[k] = sh[lane * S + k];
#pragma unroll
      for (int m = 32; m < kSumSlices; m += 32) t4[k] = t4[k] + sh[(lane + m) * S + k];
    }
    const double t = warp_sums<S>(t4, lane);
    if (sum_lane<S>(lane)) a.partials[chunk * S + comp] = t;
  }
}

struct SumsFinish {
  const double* partials;
  int nchunks;
  double* totals;
};
template <int S>
__global__ void __launch_bounds__(FV_NT) sums_finish_kernel(SumsFinish a) {
  __shared__ double sh[FV_NT * S];
  grid_dep_wait();
  grid_dep_launch();
  double acc[S];
#pragma unroll
  for (int k = 0; k < S; ++k) acc[k] = 0.0;
  for (int c = threadIdx.x; c < a.nchunks; c += FV_NT) {
#pragma unroll
    for (int k = 0; k < S; ++k) acc[k] = acc[k] + a.partials[(int64_t)c * S + k];
  }
  block_sum_fixed<S>(acc, sh);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < S; ++k) a.totals[k] = acc[k];
  }
}

template <typename T, int D>
static cudaError_t launch_sums_t(const fv_batch* h, const SumLaunch& l, int nchunks) {
  SumParams<T> a;
  a.q = static_cast<const T*>(l.q);
  a.off = l.off;
  a.sizes = l.sizes;
  a.n = l.n;
  a.halo = l.halo;
  a.pmax = h->max_patch_size;
  a.partials = l.partials;
  a.status = l.status;
  a.per_patch = l.per_patch;
  if (nchunks <= kSumFewChunks)
    return launch_kernel(sums_kernel<T, D, 512>, nchunks * kSumCluster, 512, 0, h->stream,
                         starts_early(h, nchunks * kSumCluster, 512), a);
  return launch_kernel(sums_kernel<T, D, 128>, nchunks * kSumCluster, 128, 0, h->stream, false, a);
}

cudaError_t launch_sums(const fv_batch* h, const SumLaunch& l, int nchunks) {
  if (h->prec == FV_FP64) {
    if (h->d == 1) return launch_sums_t<double, 1>(h, l, nchunks);
    if (h->d == 2) return launch_sums_t<double, 2>(h, l, nchunks);
    return launch_sums_t<double, 3>(h, l, nchunks);
  }
  if (h->d == 1) return launch_sums_t<float, 1>(h, l, nchunks);
  if (h->d == 2) return launch_sums_t<float, 2>(h, l, nchunks);
  return launch_sums_t<float, 3>(h, l, nchunks);
}

cudaError_t launch_sums_finish(const fv_batch* h, const double* partials, int nchunks,
                               double* totals) {
  const SumsFinish a{partials, nchunks, totals};
  if (h->d == 1) return launch_kernel(sums_finish_kernel<3>, 1, FV_NT, 0, h->stream, true, a);
  if (h->d == 2) return launch_kernel(sums_finish_kernel<4>, 1, FV_NT, 0, h->stream, true, a);
  return launch_kernel(sums_finish_kernel<5>, 1, FV_NT, 0, h->stream, true, a);
}

// ---------------------------------------------------------------------------
// One 64-bit word set to zero on the stream (the wave-speed slot a time step
// accumulates into, the work-queue counter), by a one-thread kernel.
// ---------------------------------------------------------------------------
__global__ void zero_word_kernel(unsigned long long* p) {
  grid_dep_wait();
  grid_dep_launch();
  *p = 0ull;
}

cudaError_t launch_zero_word(unsigned long long* p, cudaStream_t stream) {
  return launch_kernel(zero_word_kernel, 1, 1, 0, stream, true, p);
}

// ---------------------------------------------------------------------------
// Self-test of the FP64 reciprocal and square root used by the kernels.
// ---------------------------------------------------------------------------
__global__ void selftest_math_kernel(const double* x, double* out, int64_t n, int which) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = which == 0 ? recip(x[i]) : sqrt_t(x[i]);
}

cudaError_t launch_selftest_math(const double* x, double* out, int64_t n, int which) {
  int64_t blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  selftest_math_kernel<<<(int)blocks, 256>>>(x, out, n, which);
  return cudaGetLastError();
}

}  // namespace fv
