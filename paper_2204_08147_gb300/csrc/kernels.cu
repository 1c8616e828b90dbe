// CUDA kernels of the estimator's hot path (sm_103a).
//
//   k_init_block   the starting block V = [I_s (x) |v_l>]_l (Sec. 3.1, eq. trace_est)
//                  from the counter-based generator (SplitMix64 on a counter)
//   k_spmm         Z = (H W_j) M_j + W_{j-1} Cp_j: the matrix-free spin-Hamiltonian
//                  block SpMM (eq. Ht) fused with the first line of Algorithm 1's
//                  loop, and the partial sums of W_j^T Z for A_j
//   k_orth         W_{j+1} = Z + W_j Cw_j (Algorithm 1, Z - Q_j A_j) with the
//                  partial sums of W_{j+1}^T W_{j+1} for the QR (pass 1), or the
//                  accumulation psi_beta += W_{j+1} E_{j+1,beta} (pass 2)
//   k_small_a/b    per bath vector, float64: A_j, Cholesky QR with breakdown
//                  deflation, the next step's mixing coefficients
//   k_gram_rows    psi = sum_j W_j E_j from the stored basis and its bath-traced Gram
//                  psi_l^T psi_l per bath vector, all betas (k_final_gram: of a given psi;
//                  k_gram_stored: the layouts k_gram_rows does not take)
//   k_pass1_cluster / k_pass1_packed   the whole first pass of the items of a batch
//
// The Krylov block of every bath vector l is never normalised in memory: the
// stored W_j relates to the orthonormal Q_j of Algorithm 1 by Q_j = W_j M_j with
// a d_s x d_s matrix M_j (the inverse Cholesky factor), applied on the fly.
// Reductions are deterministic: per-thread partial sums, a fixed-order block
// reduction into per-block partials, and a fixed-order sum over blocks.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <array>
#include <map>
#include <mutex>
#include <set>
#include <type_traits>
#include <vector>

#include "rdm_internal.h"

namespace rdm {
namespace {

__device__ __forceinline__ uint64_t splitmix64(uint64_t seed, uint64_t n) {
  uint64_t z = seed + n * 0x9E3779B97F4A7C15ull;
  z ^= z >> 30;
  z *= 0xBF58476D1CE4E5B9ull;
  z ^= z >> 27;
  z *= 0x94D049BB133111EBull;
  z ^= z >> 31;
  return z;
}

__device__ __forceinline__ double gauss_raw(uint64_t seed, uint64_t l, uint64_t b) {
  const uint64_t base = l << 40;
  const uint64_t z1 = splitmix64(seed, (base | (2 * b)) + 1);
  const uint64_t z2 = splitmix64(seed, (base | (2 * b + 1)) + 1);
  const double u1 = ((double)(z1 >> 11) + 0.5) * 0x1.0p-53;
  const double u2 = ((double)(z2 >> 11) + 0.5) * 0x1.0p-53;
  return sqrt(-2.0 * log(u1)) * cos(2.0 * 3.141592653589793 * u2);
}

// ---- VW-wide vector access (VW * sizeof(T) is 8, 16 or 32 bytes).
template <typename T, int VW>
struct VecIO;
template <>
struct VecIO<float, 4> {
  __device__ static void st_cs(float* p, const float* r) {  // streaming (evict-first) store
    __stcs(reinterpret_cast<float4*>(p), make_float4(r[0], r[1], r[2], r[3]));
  }
  __device__ static void ld(float* r, const float* p) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
  }
  __device__ static void ld_rw(float* r, const float* p) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
  }
  __device__ static void st(float* p, const float* r) {
    *reinterpret_cast<float4*>(p) = make_float4(r[0], r[1], r[2], r[3]);
  }
};
template <>
struct VecIO<double, 2> {
  __device__ static void st_cs(double* p, const double* r) {
    __stcs(reinterpret_cast<double2*>(p), make_double2(r[0], r[1]));
  }
  __device__ static void ld(double* r, const double* p) {
    const double2 v = __ldg(reinterpret_cast<const double2*>(p));
    r[0] = v.x; r[1] = v.y;
  }
  __device__ static void ld_rw(double* r, const double* p) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    r[0] = v.x; r[1] = v.y;
  }
  __device__ static void st(double* p, const double* r) {
    *reinterpret_cast<double2*>(p) = make_double2(r[0], r[1]);
  }
};
template <>
struct VecIO<double, 4> {
  __device__ static void st_cs(double* p, const double* r) {
    VecIO<double, 2>::st_cs(p, r);
    VecIO<double, 2>::st_cs(p + 2, r + 2);
  }
  __device__ static void ld(double* r, const double* p) {
    VecIO<double, 2>::ld(r, p);
    VecIO<double, 2>::ld(r + 2, p + 2);
  }
  __device__ static void ld_rw(double* r, const double* p) {
    VecIO<double, 2>::ld_rw(r, p);
    VecIO<double, 2>::ld_rw(r + 2, p + 2);
  }
  __device__ static void st(double* p, const double* r) {
    VecIO<double, 2>::st(p, r);
    VecIO<double, 2>::st(p + 2, r + 2);
  }
};

// Mask of the lanes of this thread's row group inside its warp.
__device__ __forceinline__ unsigned group_mask(int tpr) {
  if (tpr >= 32) return 0xffffffffu;
  const unsigned lane = threadIdx.x & 31u;
  return ((1u << tpr) - 1u) << (lane & ~(unsigned)(tpr - 1));
}

// Sums held as an unevaluated pair hi + lo of floats (Knuth's two-sum): the float32 kernels'
// long sums, off the narrow float64 pipe.
struct Pair32 {
  float hi = 0.0f, lo = 0.0f;
  __device__ __forceinline__ void add(float x) {
    const float s = __fadd_rn(hi, x), t = __fsub_rn(s, hi);
    lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, t)), __fsub_rn(x, t)));
    hi = s;
  }
  __device__ __forceinline__ void add(const Pair32& o) {
    add(o.hi);
    lo = __fadd_rn(lo, o.lo);
  }
  __device__ __forceinline__ double value() const { return (double)hi + (double)lo; }
};
__device__ __forceinline__ Pair32 shfl_xor(const Pair32& p, int o) {
  Pair32 r;
  r.hi = __shfl_xor_sync(0xffffffffu, p.hi, o);
  r.lo = __shfl_xor_sync(0xffffffffu, p.lo, o);
  return r;
}
__device__ __forceinline__ float shfl_xor(float x, int o) { return __shfl_xor_sync(0xffffffffu, x, o); }
__device__ __forceinline__ void add_to(float& x, float y) { x += y; }
__device__ __forceinline__ void add_to(Pair32& x, const Pair32& y) { x.add(y); }

// The sums over the 16 lanes of one parity of a warp of NV (4, 8 or 16) values, a fixed tree
// whose every level halves the values a lane still holds (NV - 1 exchanges instead of 4 NV):
// each lane returns one, number warp_sum_index<NV>().
template <int NV, typename P>
__device__ __forceinline__ P warp_sum(P (&v)[NV]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int l = 0; l < 4; ++l) {
    const int o = 16 >> l, half = NV >> (l + 1);
    if (half == 0) {
      add_to(v[0], shfl_xor(v[0], o));
      continue;
    }
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < NV / 2; ++i) {
      if (i >= half) break;
      const P keep = up ? v[i + half] : v[i], send = up ? v[i] : v[i + half];
      v[i] = keep;
      add_to(v[i], shfl_xor(send, o));
    }
  }
  return v[0];
}
template <int NV>
__device__ __forceinline__ int warp_sum_index() {
  static_assert(NV == 4 || NV == 8 || NV == 16, "values of a 16-byte lane");
  return (int)(threadIdx.x & 31) >> (NV == 16 ? 1 : NV == 8 ? 2 : 3);
}
// One of the lanes that hold the same sum (NV < 16).
template <int NV>
__device__ __forceinline__ bool warp_sum_writes() {
  return ((threadIdx.x & 31) & (NV == 16 ? 0 : NV == 8 ? 2 : 6)) == 0;
}

// Fixed-order block reduction of NV values per thread into per-block float64
// partials: partials[((slice*gridx + bx)*G_s + lane*NG + g)*NVG + v] where
// vals[g*NVG + v] belongs to group g of the thread and lane = threadIdx.x % tpr
// (tpr <= 8, a power of two), slot = slice*gridx + bx the block's place in the grid
// (blockIdx.y * gridDim.x + blockIdx.x for a plain launch). A butterfly over the lanes of a warp with the same
// lane in the type R of vals, then the warps' sums added in float64 in warp order:
// the same order on every run. The float32 path runs the butterfly in float32 (its
// per-thread sums are float32 already): GB300's float64 pipe is narrow, and a float64
// butterfly in every block made launches of many short blocks float64-bound.
template <int NG, int NVG, typename R = double>
__device__ void block_reduce_store(const R* vals, int tpr, double* partials, int gs, size_t slot) {
  constexpr int NV = NG * NVG;
  constexpr int kWarps = kThreads / 32;
  __shared__ double red[kWarps * 8 * NV];
  const int warp = threadIdx.x >> 5, wl = threadIdx.x & 31;
  R v[NV];
#pragma unroll
  for (int e = 0; e < NV; ++e) {
    R x = vals[e];
    for (int o = tpr; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    v[e] = x;
  }
  if (wl < tpr) {
#pragma unroll
    for (int e = 0; e < NV; ++e) red[(warp * tpr + wl) * NV + e] = (double)v[e];
  }
  __syncthreads();
  if ((int)threadIdx.x < tpr * NV) {
    const int lane = threadIdx.x / NV, e = threadIdx.x % NV;
    double sum = 0.0;
    for (int w = 0; w < kWarps; ++w) sum += red[(w * tpr + lane) * NV + e];
    const size_t base = (slot * gs + (size_t)lane * NG) * NVG;
    partials[base + e] = sum;
  }
}

// The block's partials (as block_reduce_store, tpr = 2) from the warps' sums: one per lane,
// number warp_sum_index of its column chunk.
template <int NV>
__device__ void warp_sums_store(const Pair32& sum, double* partials, size_t slot) {
  constexpr int kWarps = kThreads / 32;
  __shared__ double red[kWarps][2 * NV];
  if (warp_sum_writes<NV>()) red[threadIdx.x >> 5][(threadIdx.x & 1) * NV + warp_sum_index<NV>()] = sum.value();
  __syncthreads();
  if (threadIdx.x < 2 * NV) {
    double s = 0.0;
    for (int w = 0; w < kWarps; ++w) s += red[w][threadIdx.x];
    partials[slot * 2 * NV + threadIdx.x] = s;
  }
}

// ---------------------------------------------------------------- init

__global__ void k_gauss_sumsq(int64_t d_b, uint64_t seed, int64_t l0, double* part, double* graw) {
  __shared__ double sh[kThreads];
  const int l = blockIdx.y;
  const int64_t chunk = (d_b + gridDim.x - 1) / gridDim.x;
  const int64_t lo = (int64_t)blockIdx.x * chunk;
  const int64_t hi = lo + chunk < d_b ? lo + chunk : d_b;
  double acc = 0.0;
  for (int64_t b = lo + threadIdx.x; b < hi; b += blockDim.x) {
    const double g = gauss_raw(seed, (uint64_t)(l0 + l), (uint64_t)b);
    if (graw) graw[(size_t)l * d_b + b] = g;
    acc += g * g;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int w = kThreads / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[(size_t)l * gridDim.x + blockIdx.x] = sh[0];
}

__global__ void k_gauss_finish(int n_v, int gx, const double* part, double* inv_norm) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= n_v) return;
  double s = 0.0;
  for (int i = 0; i < gx; ++i) s += part[(size_t)l * gx + i];
  inv_norm[l] = 1.0 / sqrt(s);
}

template <typename T, int DS, int VW>
__global__ void __launch_bounds__(kThreads) k_init_block(Layout L, int dist, uint64_t seed,
                                                         int64_t l0, int nvr, const double* inv_norm,
                                                         const T* vbuf, T* W, int sub, BathPerm bp) {
  constexpr int NG = VW / DS;
  const int tpr = L.TPR, rpb = kThreads / tpr;
  const int lane = threadIdx.x % tpr, rs = threadIdx.x / tpr;
  const int slice = blockIdx.y;
  T* base = W + (size_t)slice * L.D * L.Bs + lane * VW;
  const int g0 = (slice * L.Bs + lane * VW) / DS;
  const uint64_t bmask = (1ull << L.n_bath_bits) - 1ull;
  const double rad = 1.0 / sqrt((double)(1ull << L.n_bath_bits));
  for (int64_t s = (int64_t)blockIdx.x * rpb + rs; s < L.D; s += (int64_t)gridDim.x * rpb) {
    const int i = (int)(s >> L.n_bath_bits);
    uint64_t b = (uint64_t)s & bmask;
    if (bp.n) {  // the caller's bath index of internal bath index b
      uint64_t bc = 0;
      for (int q = 0; q < bp.n; ++q) bc |= ((b >> q) & 1ull) << bp.src[q];
      b = bc;
    }
    T v[VW];
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      // group g0 + g: bath vector l, system index ic of its column when the groups are
      // single columns of sub-column bath vectors (per-column recurrences), else 0
      const int l = (g0 + g) / sub, ic = (g0 + g) % sub;
      double val = 0.0;
      if (l < nvr) {
        const uint64_t lg = (uint64_t)(l0 + l);  // index in the seeded sequence
        if (dist == RDM_RADEMACHER) {
          const uint64_t z = splitmix64(seed, ((lg << 40) | b) + 1);
          val = (z >> 63) ? -rad : rad;
        } else if (dist == RDM_GAUSS) {
          val = inv_norm ? gauss_raw(seed, lg, b) * inv_norm[l]
                         : (double)vbuf[((size_t)l << L.n_bath_bits) + b];
        } else {
          val = (b == lg) ? 1.0 : 0.0;
        }
      }
#pragma unroll
      for (int a = 0; a < DS; ++a) v[g * DS + a] = (a + ic == i) ? (T)val : (T)0;
    }
    VecIO<T, VW>::st(base + (size_t)s * L.Bs, v);
  }
}

__global__ void k_gauss_fill(int64_t d_b, uint64_t seed, int64_t l0, const double* inv_norm,
                             const double* graw, int precision, void* vbuf) {
  const int l = blockIdx.y;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < d_b;
       b += (int64_t)gridDim.x * blockDim.x) {
    const double g = graw ? graw[(size_t)l * d_b + b] : gauss_raw(seed, (uint64_t)(l0 + l), (uint64_t)b);
    const double v = g * inv_norm[l];
    if (precision == RDM_FP32)
      reinterpret_cast<float*>(vbuf)[(size_t)l * d_b + b] = (float)v;
    else
      reinterpret_cast<double*>(vbuf)[(size_t)l * d_b + b] = v;
  }
}

// A table of the tiled diagonal (TileDiag): one block per tile (grid stride). The block
// first sums K_0 .. K_G of the tile (float64, shared memory), then thread rg writes
// A_q(tile, rg) of every row-group-dependent character q and thread 0 the others.
template <typename T>
__global__ void __launch_bounds__(kThreads) k_tile_diag(int64_t tiles, TileDiag dg, int stride, T* out) {
  extern __shared__ __align__(16) unsigned char smem_k[];
  double* sK = reinterpret_cast<double*>(smem_k);  // [G + 1]
  constexpr int kRG = 1 << kTileRegShift;
  for (int64_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint32_t ut = (uint32_t)t;
    for (int g = threadIdx.x; g <= dg.n_groups; g += blockDim.x) {
      double k = 0.0;
      for (int i = dg.slot_start[g]; i < dg.slot_start[g + 1]; ++i)
        k += (__popc(ut & dg.thi[i]) & 1) ? -dg.tc[i] : dg.tc[i];
      sK[g] = k;
    }
    __syncthreads();
    T* o = out + t * stride;
    for (int rg = threadIdx.x; rg < kRG; rg += blockDim.x) {
      for (int q = 0; q < 8; ++q) {
        const bool dep = (dg.dep >> q) & 1u;
        if (!dep && rg != 0) continue;
        double a = q == 0 ? sK[0] : 0.0;
        for (int g = dg.hstart[q]; g < dg.hstart[q + 1]; ++g)
          a += (__popc((uint32_t)rg & dg.mlo[g]) & 1) ? -sK[1 + g] : sK[1 + g];
        o[dg.off[q] + (dep ? rg : 0)] = (T)a;
      }
    }
    for (int e = dg.n_entries + threadIdx.x; e < stride; e += blockDim.x) o[e] = (T)0;
    __syncthreads();
  }
}

// ---------------------------------------------------------------- SpMM step

template <typename T>
struct TermsSmem {
  uint32_t* fmask;
  T* fodd;
  T* feven;
  uint32_t* dmask;
  T* dc;
};

template <typename T>
__device__ TermsSmem<T> load_terms(const FlipTerm* flips, int nf, const DiagTerm* diags, int nd) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  TermsSmem<T> t;
  T* tp = reinterpret_cast<T*>(smem_raw);
  t.fodd = tp;
  t.feven = tp + nf;
  t.dc = tp + 2 * nf;
  uint32_t* up = reinterpret_cast<uint32_t*>(tp + 2 * nf + nd);
  t.fmask = up;
  t.dmask = up + nf;
  for (int i = threadIdx.x; i < nf; i += blockDim.x) {
    t.fmask[i] = flips[i].mask;
    t.fodd[i] = (T)flips[i].c_odd;
    t.feven[i] = (T)flips[i].c_even;
  }
  for (int i = threadIdx.x; i < nd; i += blockDim.x) {
    t.dmask[i] = diags[i].mask;
    t.dc[i] = (T)diags[i].c;
  }
  __syncthreads();
  return t;
}

// The rows of block (bx, by) of a grid of gx x n_slices blocks of the untiled SpMM:
// rows bx*rpb + rs + i*gx*rpb of slice by (the grid-stride walk of a plain launch), and,
// in pass 1, its partial sums of W_j^T Z at slot by*gx + bx. `terms` are the term tables
// in shared memory (load_terms).
template <typename T, int VW, bool COH>
__device__ __forceinline__ void ld_vec(T* r, const T* p) {
  if constexpr (COH)
    VecIO<T, VW>::ld_rw(r, p);
  else
    VecIO<T, VW>::ld(r, p);
}

// COH: coherent loads only (no read-only cache path), for blocks written earlier in the
// same launch (the packed kernel).
template <typename T, int DS, int VW, int MODE, bool COH = false>
__device__ __forceinline__ void spmm_block(const Layout& L, const SpmmArgs& a, const TermsSmem<T>& terms,
                                           int bx, int by, int gx) {
  constexpr int NG = VW / DS;
  constexpr int NVG = DS * DS;
  const int tpr = L.TPR, rpb = kThreads / tpr;
  const int lane = threadIdx.x % tpr, rs = threadIdx.x / tpr;
  const int slice = by;
  const size_t soff = (size_t)slice * L.D * L.Bs + (size_t)lane * VW;
  const T* __restrict__ W = reinterpret_cast<const T*>(a.w) + soff;
  const T* __restrict__ Wp = a.w_prev ? reinterpret_cast<const T*>(a.w_prev) + soff : nullptr;
  T* __restrict__ Z = reinterpret_cast<T*>(a.z) + soff;
  const int g0 = (slice * L.Bs + lane * VW) / DS;
  const unsigned gmask = group_mask(tpr);

  T mz[NG][DS][DS], cp[NG][DS][DS];
  if (MODE != kModeApply) {
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < DS; ++i)
#pragma unroll
        for (int j = 0; j < DS; ++j) {
          mz[g][i][j] = (T)a.mz[(size_t)(g0 + g) * NVG + i * DS + j];
          cp[g][i][j] = Wp ? (T)a.cp[(size_t)(g0 + g) * NVG + i * DS + j] : (T)0;
        }
  }
  T acc[NG][DS][DS];
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int i = 0; i < DS; ++i)
#pragma unroll
      for (int j = 0; j < DS; ++j) acc[g][i][j] = (T)0;

  const int nf = a.n_flip, nd = a.n_diag;
  for (int64_t s = (int64_t)bx * rpb + rs; s < L.D; s += (int64_t)gx * rpb) {
    const uint32_t su = (uint32_t)s;
    T x[VW];
    ld_vec<T, VW, COH>(x, W + (size_t)s * L.Bs);
    // Diagonal: sum_t c_t (1 - 2 parity(s & m_t)), split over the row group.
    T dg = (T)0;
    for (int t = lane; t < nd; t += tpr) {
      const T c = terms.dc[t];
      dg += (__popc(su & terms.dmask[t]) & 1) ? -c : c;
    }
    for (int off = tpr >> 1; off > 0; off >>= 1) dg += __shfl_xor_sync(gmask, dg, off, tpr);
    T y[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) y[v] = dg * x[v];
    // Off-diagonal: y += c(parity(s & m)) x[s ^ m].
    for (int t = 0; t < nf; ++t) {
      const uint32_t m = terms.fmask[t];
      const T c = (__popc(su & m) & 1) ? terms.fodd[t] : terms.feven[t];
      if (c != (T)0) {
        T xp[VW];
        ld_vec<T, VW, COH>(xp, W + (size_t)(su ^ m) * L.Bs);
#pragma unroll
        for (int v = 0; v < VW; ++v) y[v] = fma(c, xp[v], y[v]);
      }
    }
    if (MODE == kModeApply) {
      VecIO<T, VW>::st(Z + (size_t)s * L.Bs, y);
      continue;
    }
    T z[VW];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int j = 0; j < DS; ++j) {
        T t = (T)0;
#pragma unroll
        for (int i = 0; i < DS; ++i) t = fma(y[g * DS + i], mz[g][i][j], t);
        z[g * DS + j] = t;
      }
    if (Wp) {
      T xp[VW];
      ld_vec<T, VW, COH>(xp, Wp + (size_t)s * L.Bs);
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int j = 0; j < DS; ++j) {
          T t = z[g * DS + j];
#pragma unroll
          for (int i = 0; i < DS; ++i) t = fma(xp[g * DS + i], cp[g][i][j], t);
          z[g * DS + j] = t;
        }
    }
    VecIO<T, VW>::st(Z + (size_t)s * L.Bs, z);
    if (MODE == kModePass1) {
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int i = 0; i < DS; ++i)
#pragma unroll
          for (int j = 0; j < DS; ++j) acc[g][i][j] = fma(x[g * DS + i], z[g * DS + j], acc[g][i][j]);
    }
  }
  if (MODE == kModePass1) {
    T vals[NG * NVG];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < DS; ++i)
#pragma unroll
        for (int j = 0; j < DS; ++j) vals[g * NVG + i * DS + j] = acc[g][i][j];
    block_reduce_store<NG, NVG, T>(vals, tpr, a.partials, L.groups_per_slice(), (size_t)by * gx + bx);
  }
}

template <typename T, int DS, int VW, int MODE>
__global__ void __launch_bounds__(kThreads) k_spmm(Layout L, SpmmArgs a) {
  const TermsSmem<T> terms = load_terms<T>(a.flips, a.n_flip, a.diags, a.n_diag);
  spmm_block<T, DS, VW, MODE>(L, a, terms, blockIdx.x, blockIdx.y, gridDim.x);
}

// ---------------------------------------------------------------- tiled SpMM
//
// Same result as k_spmm, organised around tiles of 2^kTileBits consecutive states of
// one slice (32 KB) held in shared memory. The own tile and, one after another, every
// partner tile tile ^ m_high that an active term needs are fetched with TMA bulk
// copies (cp.async.bulk, completion on an mbarrier) through a ring of slots, so later
// tiles stream in while the current one is consumed. Every flip term is then a
// shared-memory (or register) read; the diagonal is rebuilt per tile from a small
// table (TileDiag). The blocks walk the (slice, tile) pairs with one grid stride,
// slice by slice, so all SMs work on neighbouring tiles of one slice and partner
// tiles are mostly served from L2.

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// Bulk copy with an L2 eviction-priority policy (createpolicy value).
__device__ __forceinline__ void bulk_load_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                               uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, "
      "[%3], %4;\n" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;\n" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
  return p;
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Producer/consumer layout of the tiled SpMM: warps 8 and 9 issue TMA bulk copies
// into a ring of shared-memory slots; the consumer warps read them. A slot holds one
// 32 KB tile (kTileRows rows of a slice) plus, for the own tile, its row of the K
// table of the diagonal. Per tile the stage sequence is: own tile, each needed partner
// tile, then the W_{j-1} tile (if any). Full barriers (count 1, transaction bytes)
// and empty barriers (one arrival per consumer warp) order the ring.
//
// What bounds it: shared memory, whose 128 bytes per clock serve both the copies and the
// consumers' 16-byte loads (ncu: loads 66% + copies 25% of the clocks for long-range XXZ
// N = 22, 57% + 35% for the transverse field), and for the transverse field the copies out
// of L2 (12.9 of the copy probe's 15.7 TB/s). Before, the consumers' instructions did:
// 20 k per warp and XXZ tile, most of them scans over the patterns, address XORs and
// per-term branches. Now the producers say with each stage what it is (ballots over the
// patterns), every term is one address and constant offsets, the parity of a thread's rows
// is a bit mask made once, and one set of loads serves all hops of a spin with the register
// spins. Per launch, before and after: long-range XXZ N = 22 (n_v = 16) 4.17 -> 2.74 ms, N = 24
// (n_v = 4) 4.95 -> 3.20 ms; long-range XY N = 16 (n_v = 400) 2.38 -> 1.38 ms (with the runs of
// tiled_run_log); ladder N = 20 (n_v = 50) 1.58 -> 1.09 ms; transverse field N = 22 (n_v = 32)
// 2.47 -> 2.38 ms.
constexpr int kConsumerWarps = (kTileRows >> kTileRegBits) * kTiledLanes / 32;
constexpr int kProducerWarps = 2;  // each issues the copies of every other ring slot
constexpr int kTiledThreads = (kConsumerWarps + kProducerWarps) * 32;
constexpr uint32_t kTileBytes = (uint32_t)kTileRows * kTiledLanes * 16;  // 32 KB
constexpr int kMaxStages = 8;
// Slot = tile + the A-table row of the diagonal (rounded to 128 bytes).
__host__ __device__ inline uint32_t tiled_slot_bytes(int n_entries, int elem) {
  return kTileBytes + ((uint32_t)(tile_diag_stride(n_entries, elem) * elem) + 127u) / 128u * 128u;
}

// Shared-memory records of the tiled SpMM's term tables (TiledTerms), in T.
template <typename T>
struct alignas(16) PatS {  // a partner pattern
  uint32_t high;   // the partner tile is tile ^ high
  uint32_t flags;  // kPatField, kPatReg
  int start, end;  // its lane terms
  T cf;            // field on its one high spin
  T co[3], ce[3];  // hops with the spins of the register rows
};
template <typename T>
struct alignas(16) LaneS {  // a term whose in-tile part moves the row group rg
  T co, ce;
  uint32_t off;  // element offset of m_low (XORed into a thread's row offset)
  uint32_t low;  // m_low
};
template <typename T>
struct alignas(16) GrpS {  // in-tile terms of one row-group spin l: field, hops with register spins
  uint32_t off, low, flags;
  T cf;
  T co[3], ce[3];
};
// What the producer says of a ring stage: the own tile's holds its index and the number
// of the tile's partner stages, a partner stage's its pattern (+ kJoint for the first of an
// opposite-spin pair) and, for a flat pattern, its coefficient in this tile.
template <typename T>
struct alignas(16) StageS {
  int what;
  uint32_t tile;  // the own tile's index
  T c;
};
constexpr int kJoint = 1 << 16;

template <typename T>
__host__ __device__ inline size_t tiled_smem_bytes(int n_part, int n_lane, int n_grp, int n_entries, int stages) {
  size_t off = (size_t)stages * tiled_slot_bytes(n_entries, (int)sizeof(T));
  off += 2 * kMaxStages * 8 + 64;                  // full/empty barriers, control
  off += 2 * 8 * 16 * sizeof(T);                   // mixing coefficients of the lanes
  off += (size_t)kConsumerWarps * kTiledLanes * 16 * 8;  // reduction scratch
  off = (off + 15) / 16 * 16;
  off += kMaxStages * sizeof(StageS<T>);
  off += (size_t)n_part * sizeof(PatS<T>);
  off += (size_t)n_grp * sizeof(GrpS<T>);
  off += (size_t)n_lane * sizeof(LaneS<T>);
  off += 16 * sizeof(T);                           // hops and fields of the register rows
  off += (size_t)kTileRows * sizeof(T);            // low table of the diagonal
  return off + 64;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(smem_u32(bar)) : "memory");
}
// Named barrier over the consumer warps with an OR of `pred` (bar.red.or).
__device__ __forceinline__ bool consumers_sync_or(bool pred) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)pred), "n"(kConsumerWarps * 32)
      : "memory");
  return r != 0;
}
// Bounded wait that also gives up when another thread has raised the abort flag.
__device__ __forceinline__ bool ring_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag) {
  for (uint32_t it = 0; it < (1u << 22); ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 255u && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}

// At a producer's end: no copy of its may still be on its way into the ring when the block
// ends. In a whole run the consumers have waited for all of them, but not after a wait that
// gave up, so it waits for the last copy into each of its slots (q, q + kProducerWarps, ..),
// bounded, and not cut short by the abort flag. slot, round: the stage after its last; the
// stage at which it stopped was not issued. (Apart: inlined, the loop cost the transverse
// field at N = 22 0.3%.)
__device__ __noinline__ void drain_ring(uint64_t* full, int stages, int q, int slot, uint32_t round, bool stop) {
  const int failed = !stop ? -1 : (slot == 0 ? stages : slot) - 1;
  for (int sl = q; sl < stages; sl += kProducerWarps) {
    const uint32_t copies = round + (sl < slot ? 1u : 0u) - (sl == failed ? 1u : 0u);
    for (uint32_t it = 0; copies && it < (1u << 20) && !mbar_try_wait(&full[sl], (copies - 1u) & 1u); ++it) {
    }
  }
}

// Rows of a consumer thread: row rg + RG m (m = 0..RPT-1) of a tile sits at element offset
// rgoff + m * kStep (rgoff = rg * BS + lane * VW, kStep = RG * BS). Under a mask m_low in the
// row-group bits its partner rows sit at (rgoff ^ m_low * BS) + m * kStep: one address and
// constant offsets. A mask bit in the register rows only renames m.
template <int STEP, typename T, int VW, int RPT>
__device__ __forceinline__ void load_rows(T (&x)[RPT][VW], const T* p) {
#pragma unroll
  for (int m = 0; m < RPT; ++m) VecIO<T, VW>::ld_rw(x[m], p + m * STEP);
}
// y += c x; float32 two columns at a time (fma.rn.f32x2 rounds each as fmaf does; few-term
// models 5% faster, but the flat partner tiles below 1.5% slower)
template <typename T, int VW>
__device__ __forceinline__ void axpy(T (&y)[VW], T c, const T (&x)[VW]) {
  if constexpr (sizeof(T) == 4) {
#pragma unroll
    for (int v = 0; v < VW; v += 2)
      asm("{\n .reg .b64 c, x, y;\n mov.b64 c, {%2, %2};\n mov.b64 x, {%3, %4};\n mov.b64 y, {%0, %1};\n"
          " fma.rn.f32x2 y, c, x, y;\n mov.b64 {%0, %1}, y;\n}\n"
          : "+f"(y[v]), "+f"(y[v + 1])
          : "f"(c), "f"(x[v]), "f"(x[v + 1]));
  } else {
#pragma unroll
    for (int v = 0; v < VW; ++v) y[v] = fma(c, x[v], y[v]);
  }
}
// Whether a coefficient is not +0, by its bits (a float64 compare would take the narrow
// float64 pipe).
__device__ __forceinline__ bool in_use(float c) { return __float_as_int(c) != 0; }
__device__ __forceinline__ bool in_use(double c) { return (__double2hiint(c) | __double2loint(c)) != 0; }
// y[m] += c * (row m of p)
template <int STEP, typename T, int VW, int RPT>
__device__ __forceinline__ void rows_fma(T (&y)[RPT][VW], const T* p, T c) {
#pragma unroll
  for (int m = 0; m < RPT; ++m) {
    T x[VW];
    VecIO<T, VW>::ld_rw(x, p + m * STEP);
    axpy(y[m], c, x);
  }
}
// y[m] += cA * (row m of a) + cB * (row m of b), the loads of both before their fmas
template <int STEP, typename T, int VW, int RPT>
__device__ __forceinline__ void rows_fma2(T (&y)[RPT][VW], const T* a, T cA, const T* b, T cB) {
#pragma unroll
  for (int m = 0; m < RPT; ++m) {
    T u[VW], w[VW];
    VecIO<T, VW>::ld_rw(u, a + m * STEP);
    VecIO<T, VW>::ld_rw(w, b + m * STEP);
#pragma unroll
    for (int v = 0; v < VW; ++v) y[m][v] = fma(cB, w[v], fma(cA, u[v], y[m][v]));
  }
}
// y[m] += c * x[m ^ K] on the rows m whose parity under K is ODD
template <int K, int ODD, typename T, int VW, int RPT>
__device__ __forceinline__ void reg_half(T (&y)[RPT][VW], const T (&x)[RPT][VW], T c) {
#pragma unroll
  for (int m = 0; m < RPT; ++m) {
    if ((((m & K) ^ ((m & K) >> 1) ^ ((m & K) >> 2)) & 1) != ODD) continue;
    axpy(y[m], c, x[m ^ K]);
  }
}
// The coefficients of both halves are the same across the warp (skipped when zero) ...
template <int K, typename T, int VW, int RPT>
__device__ __forceinline__ void reg_uniform(T (&y)[RPT][VW], const T (&x)[RPT][VW], T c_even, T c_odd) {
  if (in_use(c_even)) reg_half<K, 0>(y, x, c_even);
  if (in_use(c_odd)) reg_half<K, 1>(y, x, c_odd);
}
// Whether a thread takes part in a term whose coefficient c may differ between the lanes of
// its warp. The recurrences' lanes all do where one of them needs it (a zero coefficient on
// the others), rather than diverge. H x of a caller's x (EXACT) leaves out the rows whose
// coefficient is zero: x may hold infinities or NaN, and 0 * x would put them into rows that H
// does not couple to theirs.
template <bool EXACT, typename T>
__device__ __forceinline__ bool lane_takes(T c) {
  return EXACT ? in_use(c) : __any_sync(0xffffffffu, in_use(c)) != 0;
}
// ... or differ between its lanes.
template <int K, bool EXACT, typename T, int VW, int RPT>
__device__ __forceinline__ void reg_lanes(T (&y)[RPT][VW], const T (&x)[RPT][VW], T c_even, T c_odd) {
  if (lane_takes<EXACT>(c_even)) reg_half<K, 0>(y, x, c_even);
  if (lane_takes<EXACT>(c_odd)) reg_half<K, 1>(y, x, c_odd);
}

// The in-tile terms: y += (terms) x, xo the thread's own rows of the tile `own`.
template <bool UNI, bool EXACT, int RG, int STEP, typename T, int VW, int RPT>
__device__ __forceinline__ void own_terms(T (&y)[RPT][VW], const T (&xo)[RPT][VW], const T* own, int rgoff,
                                          const TiledTerms& tt, const T* s_reg, const GrpS<T>* grp,
                                          const LaneS<T>* lanet, uint32_t act_lane, uint32_t act_grp) {
  const uint32_t reg_flags = tt.reg_flags;
  // fields and hops of the register rows alone
  if (reg_flags & 2u) reg_uniform<1>(y, xo, s_reg[8 + 1], s_reg[1]);
  if (reg_flags & 4u) reg_uniform<2>(y, xo, s_reg[8 + 2], s_reg[2]);
  if (reg_flags & 16u) reg_uniform<4>(y, xo, s_reg[8 + 4], s_reg[4]);
  if constexpr (!UNI) {
    if (reg_flags & 8u) reg_uniform<3>(y, xo, s_reg[8 + 3], s_reg[3]);
    if (reg_flags & 32u) reg_uniform<5>(y, xo, s_reg[8 + 5], s_reg[5]);
    if (reg_flags & 64u) reg_uniform<6>(y, xo, s_reg[8 + 6], s_reg[6]);
  } else if (reg_flags & (8u | 32u | 64u)) {
    reg_uniform<3>(y, xo, s_reg[8 + 3], s_reg[3]);
    reg_uniform<5>(y, xo, s_reg[8 + 5], s_reg[5]);
    reg_uniform<6>(y, xo, s_reg[8 + 6], s_reg[6]);
  }
  // a row-group spin's field and its hops with the register spins share one set of loads
  for (int t = 0; t < tt.n_grp; ++t) {
    const GrpS<T>& G = grp[t];
    const bool odd = (act_grp >> t) & 1u;
    const uint32_t fl = G.flags;
    T xp[RPT][VW];
    load_rows<STEP>(xp, own + (rgoff ^ (int)G.off));
    if (fl & kPatField) {
      const T c = G.cf;
#pragma unroll
      for (int m = 0; m < RPT; ++m) axpy(y[m], c, xp[m]);
    }
    if (fl & kPatReg) reg_lanes<1, EXACT>(y, xp, odd ? G.co[0] : G.ce[0], odd ? G.ce[0] : G.co[0]);
    if (fl & (kPatReg << 1)) reg_lanes<2, EXACT>(y, xp, odd ? G.co[1] : G.ce[1], odd ? G.ce[1] : G.co[1]);
    if (fl & (kPatReg << 2)) reg_lanes<4, EXACT>(y, xp, odd ? G.co[2] : G.ce[2], odd ? G.ce[2] : G.co[2]);
  }
  // terms of the row-group spins alone
  if constexpr (UNI) {
    int t = 0;
    for (; t + 1 < tt.n_own; t += 2)
      rows_fma2<STEP>(y, own + (rgoff ^ (int)lanet[t].off), lanet[t].co, own + (rgoff ^ (int)lanet[t + 1].off),
                       lanet[t + 1].co);
    if (t < tt.n_own) rows_fma<STEP>(y, own + (rgoff ^ (int)lanet[t].off), lanet[t].co);
  } else {
    for (int t = 0; t < tt.n_own; ++t) {
      const LaneS<T> d = lanet[t];
      const T c = ((act_lane >> t) & 1u) ? d.co : d.ce;
      if (lane_takes<EXACT>(c)) rows_fma<STEP>(y, own + (rgoff ^ (int)d.off), c);
    }
  }
}
// The terms of one high spin on its partner tile P: its field and its hops with in-tile
// spins (hs: whether it is down here).
template <bool UNI, bool EXACT, int STEP, typename T, int VW, int RPT>
__device__ __forceinline__ void single_terms(T (&y)[RPT][VW], const T* P, int rgoff, int rg, const PatS<T>& A, bool hs,
                                             const LaneS<T>* lanet) {
  const uint32_t fl = A.flags;
  if (fl & (kPatField | (kPatReg * 7u))) {
    T xp[RPT][VW];
    load_rows<STEP>(xp, P + rgoff);
    if (fl & kPatField) {
      const T c = A.cf;
#pragma unroll
      for (int m = 0; m < RPT; ++m) axpy(y[m], c, xp[m]);
    }
    if (fl & kPatReg) reg_uniform<1>(y, xp, hs ? A.co[0] : A.ce[0], hs ? A.ce[0] : A.co[0]);
    if (fl & (kPatReg << 1)) reg_uniform<2>(y, xp, hs ? A.co[1] : A.ce[1], hs ? A.ce[1] : A.co[1]);
    if (fl & (kPatReg << 2)) reg_uniform<4>(y, xp, hs ? A.co[2] : A.ce[2], hs ? A.ce[2] : A.co[2]);
  }
  for (int t = A.start; t < A.end; ++t) {
    const LaneS<T> d = lanet[t];
    const bool odd = (((uint32_t)rg & d.low) != 0u) != hs;
    const T c = UNI || odd ? d.co : d.ce;
    if (UNI || lane_takes<EXACT>(c)) rows_fma<STEP>(y, P + (rgoff ^ (int)d.off), c);
  }
}
// An opposite-spin pair: term l of group A (its spin down here, tile Z) acts on the rows
// whose spin l is up, of group B (spin up, tile O) on the others, so every row takes exactly
// one of the two.
template <int STEP, typename T, int VW, int RPT>
__device__ __forceinline__ void pair_terms(T (&y)[RPT][VW], const T* Z, const T* O, int rgoff, int rg,
                                           const PatS<T>& A, const PatS<T>& B, const LaneS<T>* lanet) {
  const uint32_t fl = A.flags;
  if (fl & (kPatReg * 7u)) {
    T xp[RPT][VW];
    load_rows<STEP>(xp, Z + rgoff);
    if (fl & kPatReg) reg_half<1, 1>(y, xp, A.co[0]);
    if (fl & (kPatReg << 1)) reg_half<2, 1>(y, xp, A.co[1]);
    if (fl & (kPatReg << 2)) reg_half<4, 1>(y, xp, A.co[2]);
    load_rows<STEP>(xp, O + rgoff);
    if (fl & kPatReg) reg_half<1, 0>(y, xp, B.co[0]);
    if (fl & (kPatReg << 1)) reg_half<2, 0>(y, xp, B.co[1]);
    if (fl & (kPatReg << 2)) reg_half<4, 0>(y, xp, B.co[2]);
  }
  const int n = A.end - A.start;
  const LaneS<T>* const la = lanet + A.start;
  const LaneS<T>* const lb = lanet + B.start;
  for (int t = 0; t < n; ++t) {
    const bool up = ((uint32_t)rg & la[t].low) != 0u;
    rows_fma<STEP>(y, (up ? Z : O) + (rgoff ^ (int)la[t].off), up ? la[t].co : lb[t].co);
  }
}

// Diagonal of H on this thread's RPT rows rg + RG m of a tile, from the tile's A-table
// row hk (TileDiag): low[r] + sum_q A_q (-1)^popc(q & m), one RPT-point Walsh-Hadamard
// transform of the A_q.
template <typename T, int RPT, int RG>
__device__ __forceinline__ void tile_diagonal(T (&dg)[RPT], const T* low, const T* hk, int rg,
                                              const TileDiag& td) {
  static_assert(RPT == (1 << kTileRegBits) && RG == (1 << kTileRegShift), "register rows per thread");
  T A[RPT];
#pragma unroll
  for (int q = 0; q < RPT; ++q) A[q] = hk[td.off[q] + (((td.dep >> q) & 1u) ? rg : 0)];
#pragma unroll
  for (int len = 1; len < RPT; len <<= 1)
#pragma unroll
    for (int i = 0; i < RPT; ++i)
      if (!(i & len)) {
        const T u = A[i], w = A[i | len];
        A[i] = u + w;
        A[i | len] = u - w;
      }
#pragma unroll
  for (int m = 0; m < RPT; ++m) dg[m] = low[rg + RG * m] + A[m];
}

// The term tables into shared memory, by all threads of the block.
template <int BS, typename T>
__device__ __forceinline__ void load_tables(const TiledTerms& tt, PatS<T>* pat, GrpS<T>* grp, LaneS<T>* lanet, T* s_reg,
                                            T* s_low) {
  for (int i = threadIdx.x; i < tt.n_part; i += blockDim.x) {
    PatS<T> r;
    const double* c = tt.pat_coef + (size_t)i * 7;
    r.high = tt.pat_high[i];
    r.flags = tt.pat_flags[i];
    r.start = tt.pat_start[i];
    r.end = tt.pat_start[i + 1];
    r.cf = (T)c[0];
    for (int q = 0; q < 3; ++q) {
      r.co[q] = (T)c[1 + q];
      r.ce[q] = (T)c[4 + q];
    }
    pat[i] = r;
  }
  for (int i = threadIdx.x; i < tt.n_grp; i += blockDim.x) {
    GrpS<T> r;
    const double* c = tt.grp_coef + (size_t)i * 7;
    r.low = tt.grp_low[i];
    r.off = r.low * BS;
    r.flags = tt.grp_flags[i];
    r.cf = (T)c[0];
    for (int q = 0; q < 3; ++q) {
      r.co[q] = (T)c[1 + q];
      r.ce[q] = (T)c[4 + q];
    }
    grp[i] = r;
  }
  for (int i = threadIdx.x; i < tt.n_lane; i += blockDim.x) {
    LaneS<T> r;
    r.co = (T)tt.lane_coef[2 * i];
    r.ce = (T)tt.lane_coef[2 * i + 1];
    r.low = tt.lane_low[i];
    r.off = r.low * BS;
    lanet[i] = r;
  }
  for (int i = threadIdx.x; i < 16; i += blockDim.x) s_reg[i] = (T)tt.reg_coef[i];
  for (int i = threadIdx.x; i < kTileRows; i += blockDim.x) s_low[i] = (T)tt.dg.low[i];
}

// TILE_SUMS (float32, pass 1): the float32 sums of W_j^T Z end with each tile; the warp's go on
// as a pair of floats. Summed on in float32 over the runs of tiles of a slice, the rounding of
// A_j grew with them (N = 18, 100 vectors, runs of 2 tiles: 5.7e-9 to 8.7e-9 of A_1). The
// sums of a tile also leave the accumulators' registers to the partner tiles (XXZ N = 22 and
// 19, XY N = 16: 1% faster solves). Not for uniform terms without runs (long slices, every
// gridDim-th tile), whose sums stay as they were: their tiles are short, and the transverse
// field at N = 22 would take 1.5% longer.
template <typename T, int DS, int MODE, bool UNI = false, bool TILE_SUMS = false>
__global__ void __launch_bounds__(kTiledThreads, 1) k_spmm_tiled(Layout L, SpmmArgs a) {
  static_assert(!TILE_SUMS || (MODE == kModePass1 && sizeof(T) == 4), "sums of the float32 first pass");
  constexpr int VW = 16 / (int)sizeof(T);
  constexpr int LPR = kTiledLanes;          // 16-byte vectors per row
  constexpr int BS = VW * LPR;              // elements per row of a slice
  // HG: a bath-vector group is wider than one lane's 16-byte vector (float64 with
  // d_s = 4: the group is the whole 32-byte row, half in each of the row's two lanes).
  // Its mixing and partial sums then take the other lane's half by a shuffle.
  constexpr bool HG = DS > VW;
  static_assert(!HG || DS == VW * LPR, "a wide group spans exactly the lanes of a row");
  constexpr int NG = HG ? 1 : VW / DS;
  constexpr int NVG = DS * DS;
  constexpr int NV = HG ? DS * VW : NG * NVG;  // partial sums per thread
  constexpr int NVC = HG ? NVG : NV;           // mixing coefficients per lane
  constexpr int RG = kConsumerWarps * 32 / LPR;  // row groups
  constexpr int RGL = (RG >= 256) ? 8 : (RG >= 128) ? 7 : (RG >= 64) ? 6 : 5;  // log2(RG)
  constexpr int RPT = kTileRows / RG;            // rows per consumer thread
  const int kStages = a.stages;
  static_assert(RPT == (1 << kTileRegBits), "rows per consumer thread");
  static_assert((1 << RGL) == RG && RGL == kTileRegShift, "row groups are the low tile bits");
  extern __shared__ __align__(128) unsigned char smem[];
  const TiledTerms& tt = a.tiled;
  const int npart = tt.n_part, nlane = tt.n_lane, npair = tt.n_pair, nsingle = tt.n_single;
  const int hstride = tile_diag_stride(tt.dg.n_entries, (int)sizeof(T));
  const uint32_t kSlotBytes = tiled_slot_bytes(tt.dg.n_entries, (int)sizeof(T));
  unsigned char* const ring = smem;
  uint64_t* const full = reinterpret_cast<uint64_t*>(smem + (size_t)kStages * kSlotBytes);
  uint64_t* const empty = full + kMaxStages;
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(empty + kMaxStages);
  T* const s_mz = reinterpret_cast<T*>(smem + (size_t)kStages * kSlotBytes + 2 * kMaxStages * 8 + 64);
  T* const s_cp = s_mz + 8 * 16;
  double* const red = reinterpret_cast<double*>(s_cp + 8 * 16);
  size_t off = (size_t)(reinterpret_cast<unsigned char*>(red + kConsumerWarps * kTiledLanes * 16) - smem);
  off = (off + 15) / 16 * 16;
  StageS<T>* const stage = reinterpret_cast<StageS<T>*>(smem + off);
  PatS<T>* const pat = reinterpret_cast<PatS<T>*>(stage + kMaxStages);
  GrpS<T>* const grp = reinterpret_cast<GrpS<T>*>(pat + npart);
  LaneS<T>* const lanet = reinterpret_cast<LaneS<T>*>(grp + tt.n_grp);
  T* const s_reg = reinterpret_cast<T*>(lanet + nlane);  // [8] c_odd, [8] c_even
  T* const s_low = s_reg + 16;

  load_tables<BS>(tt, pat, grp, lanet, s_reg, s_low);
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kConsumerWarps);
    }
    *abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();

  const int warp = threadIdx.x >> 5;
  const int tile_log = L.n_bits - kTileBits;  // tiles per slice = 2^tile_log
  const int64_t n_tiles = (int64_t)L.n_slices << tile_log;
  const uint32_t tile_mask = (uint32_t)(((int64_t)1 << tile_log) - 1);
  const bool has_prev = a.w_prev != nullptr;
  // Tiles of a block come in runs of 2^run_log consecutive (slice, tile) places.
  const int run_log = a.run_log;
  const int64_t n_runs = n_tiles >> run_log;
  const int run_mask = (1 << run_log) - 1;

  if (warp >= kConsumerWarps) {
    // ------------------------------------------------ producers
    // Both warps walk the whole stage sequence; producer q's lane 0 issues the stages with
    // seq % kProducerWarps == q (the ring depth is a multiple of kProducerWarps, so each
    // owns fixed slots). Per tile, ballots over the patterns give the stages it needs: pairs
    // of patterns consumed together, single-spin patterns, then the others in use.
    const int pl = threadIdx.x & 31;
    const uint32_t q = (uint32_t)(warp - kConsumerWarps);
    // W_j tiles are reused as partners of neighbouring tiles: keep them in L2;
    // W_{j-1} tiles are read once: let them leave first.
    const uint64_t keep = policy_evict_last();
    const uint64_t stream = policy_evict_first();
    const uint32_t hk_bytes = (uint32_t)hstride * (uint32_t)sizeof(T);
    const T* const hk_table = reinterpret_cast<const T*>(a.tile_k);
    const int flat0 = npair + nsingle, nflat = npart - flat0;
    // stage counter kept as (slot, round) so no division by the runtime ring depth
    uint32_t seq = 0, round = 0;
    int slot = 0;
    bool stop = false;
    // Waits for the next slot if it is this producer's, has lane 0 call fill(slot address)
    // and moves on; false when a wait gave up.
    auto next_stage = [&](uint32_t ut, int what, T c, const void* src, uint32_t extra, const void* src2, uint64_t policy) {
      if (seq % kProducerWarps == q) {
        bool ok = true;
        if (pl == 0) {
          ok = round == 0 || ring_wait(&empty[slot], (round - 1u) & 1u, abort_flag);
          if (ok) {
            unsigned char* dst = ring + (size_t)slot * kSlotBytes;
            stage[slot].what = what;
            stage[slot].tile = ut;
            stage[slot].c = c;
            fence_proxy_async();
            mbar_expect_tx(&full[slot], kTileBytes + extra);
            bulk_load_hint(dst, src, kTileBytes, &full[slot], policy);
            if (extra) bulk_load_hint(dst + kTileBytes, src2, extra, &full[slot], policy);
          }
        }
        if (!__shfl_sync(0xffffffffu, (int)ok, 0)) stop = true;
      }
      ++seq;
      if (++slot == kStages) {
        slot = 0;
        ++round;
      }
    };
    for (int64_t run = blockIdx.x; run < n_runs && !stop; run += gridDim.x)
      for (int rt = 0; rt <= run_mask && !stop; ++rt) {
        const int64_t gt = (run << run_log) + rt;
        const int slice = (int)(gt >> tile_log);
        const uint32_t ut = tt.tile_order[(uint32_t)gt & tile_mask];
        const size_t soff = (size_t)slice * L.D * BS;
        const T* W = reinterpret_cast<const T*>(a.w) + soff;
        auto tile_of = [&](uint32_t t) { return W + ((size_t)t << kTileBits) * BS; };
        // pairable groups with their high spin up / down in this tile
        const bool in_pair = pl < npair;
        const bool up = in_pair && (ut & pat[pl].high) != 0u;
        uint32_t om = __ballot_sync(0xffffffffu, up), zm = __ballot_sync(0xffffffffu, in_pair && !up);
        int n_st = npair + nsingle;
        for (int f0 = 0; f0 < nflat; f0 += 32) {
          bool on = false;
          if (f0 + pl < nflat) {
            const PatS<T>& A = pat[flat0 + f0 + pl];
            on = in_use((__popc(ut & A.high) & 1) ? A.co[0] : A.ce[0]);
          }
          n_st += __popc(__ballot_sync(0xffffffffu, on));
        }
        next_stage(ut, n_st, (T)0, tile_of(ut), hk_bytes, hk_table + (size_t)ut * hstride, keep);
        for (int joint = __popc(zm) < __popc(om) ? __popc(zm) : __popc(om); (zm | om) && !stop; --joint) {
          // down and up groups alternate, then the rest of the longer list
          if (joint > 0) {
            const int z = __ffs((int)zm) - 1, o = __ffs((int)om) - 1;
            zm &= zm - 1u;
            om &= om - 1u;
            next_stage(ut, z | kJoint, (T)0, tile_of(ut ^ pat[z].high), 0u, nullptr, keep);
            if (!stop) next_stage(ut, o, (T)0, tile_of(ut ^ pat[o].high), 0u, nullptr, keep);
          } else {
            const int p = __ffs((int)(zm | om)) - 1;
            zm &= ~(1u << p);
            om &= ~(1u << p);
            next_stage(ut, p, (T)0, tile_of(ut ^ pat[p].high), 0u, nullptr, keep);
          }
        }
        for (int p = npair; p < flat0 && !stop; ++p)
          next_stage(ut, p, (T)0, tile_of(ut ^ pat[p].high), 0u, nullptr, keep);
        for (int f0 = 0; f0 < nflat && !stop; f0 += 32) {
          T c = (T)0;
          if (f0 + pl < nflat) {
            const PatS<T>& A = pat[flat0 + f0 + pl];
            c = (__popc(ut & A.high) & 1) ? A.co[0] : A.ce[0];
          }
          for (uint32_t m = __ballot_sync(0xffffffffu, in_use(c)); m && !stop; m &= m - 1u) {
            const int i = __ffs((int)m) - 1, p = flat0 + f0 + i;
            next_stage(ut, p, __shfl_sync(0xffffffffu, c, i), tile_of(ut ^ pat[p].high), 0u, nullptr, keep);
          }
        }
        if (has_prev && !stop) {
          const T* Wp = reinterpret_cast<const T*>(a.w_prev) + soff;
          next_stage(ut, 0, (T)0, Wp + ((size_t)ut << kTileBits) * BS, 0u, nullptr, stream);
        }
      }
    if (pl == 0) {
      drain_ring(full, kStages, (int)q, slot, round, stop);
      if (stop) atomicOr(a.err, 1u);
    }
    return;
  }

  // -------------------------------------------------- consumers
  const int lane = threadIdx.x % LPR;  // 16-byte column chunk of a row
  const int rg = threadIdx.x / LPR;    // row group: rows rg + RG*m
  constexpr int kStep = RG * BS;        // elements between a thread's rows
  const int rgoff = rg * BS + lane * VW;  // element offset of its first row in a tile
  const bool leader = (threadIdx.x & 31) == 0;
  // next unreleased ring stage as (slot, phase parity): no division by the runtime depth
  int rslot = 0;
  uint32_t rphase = 0;
  bool aborted = false;
  // Waits for the ring slot `ahead` (0 or 1) stages past the next unreleased one.
  int at = 0;  // the slot last waited for
  auto acquire = [&](const T*& slot_ptr, int ahead) -> bool {
    int slot = rslot + ahead;
    uint32_t ph = rphase;
    if (slot >= kStages) {
      slot -= kStages;
      ph ^= 1u;
    }
    if (!ring_wait(&full[slot], ph, abort_flag)) return false;
    slot_ptr = reinterpret_cast<const T*>(ring + (size_t)slot * kSlotBytes);
    at = slot;
    return true;
  };
  auto release = [&]() {
    __syncwarp();
    if (leader) mbar_arrive(&empty[rslot]);
    if (++rslot == kStages) {
      rslot = 0;
      rphase ^= 1u;
    }
  };
  auto release2 = [&]() {  // the next two stages
    __syncwarp();
    const int s2 = rslot + 1 == kStages ? 0 : rslot + 1;
    if (leader) {
      mbar_arrive(&empty[rslot]);
      mbar_arrive(&empty[s2]);
    }
    if (s2 < rslot) rphase ^= 1u;
    rslot = s2 + 1;
    if (rslot == kStages) {
      rslot = 0;
      rphase ^= 1u;
    }
  };
  // Partials of W_j^T Z of this block for one slice (zero for a slice it has no tile
  // of); every (slice, block) entry is written once.
  const int gs = BS / DS;
  auto partial_base = [&](int slice) -> size_t {
    return ((size_t)(slice * gridDim.x + blockIdx.x) * gs + (HG ? 0 : (size_t)threadIdx.x * NG)) * NVG;
  };
  // Entry e of a lane's partial sums in its group's DS x DS block: (i, j) = (e / VW,
  // lane * VW + e % VW) for wide groups (lane = threadIdx.x here, < LPR).
  auto partial_entry = [&](int e) -> int {
    return HG ? (e / VW) * DS + (int)threadIdx.x * VW + e % VW : e;
  };

  // W_j^T Z sums of this lane's bath-vector groups, of one tile (TILE_SUMS) or of the slice
  Pair32 psum;
  T acc[NV];
#pragma unroll
  for (int e = 0; e < NV; ++e) acc[e] = (T)0;
  T* __restrict__ Z = nullptr;
  int cur = -1;       // slice of the tiles in progress
  int unwritten = 0;  // slices [unwritten, n_slices) have no partials yet
  // Parity of this thread's row group under the in-tile lane terms and groups (bit t).
  uint32_t act_lane = 0u, act_grp = 0u;
  for (int t = 0; t < tt.n_own; ++t) act_lane |= (uint32_t)(__popc((uint32_t)rg & lanet[t].low) & 1) << t;
  for (int t = 0; t < tt.n_grp; ++t) act_grp |= (uint32_t)(((uint32_t)rg & grp[t].low) != 0u) << t;

  // The consumers walk the same (slice, tile) sequence as the producers. At every
  // change of slice (and at the end) they close the finished slice; every consumer
  // thread passes the same barriers, also after an abort.
  int64_t run = blockIdx.x;
  for (int rt = 0;; ++rt) {
    if (rt > run_mask) {
      rt = 0;
      run += gridDim.x;
    }
    const int64_t gt = (run << run_log) + rt;
    const int slice = run < n_runs ? (int)(gt >> tile_log) : L.n_slices;
    if (slice != cur) {
      if (consumers_sync_or(aborted)) aborted = true;
      if (MODE == kModePass1 && !aborted) {
        if (cur >= 0) {
          // fixed-order reduction: the sums within a warp, then the warps in order in float64
          if constexpr (TILE_SUMS) {
            if (warp_sum_writes<NV>()) red[(warp * LPR + lane) * 16 + warp_sum_index<NV>()] = psum.value();
          } else {
            T v[NV];
#pragma unroll
            for (int e = 0; e < NV; ++e) {
              T x = acc[e];
#pragma unroll
              for (int o = LPR; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
              v[e] = x;
            }
            if ((threadIdx.x & 31) < LPR) {
#pragma unroll
              for (int e = 0; e < NV; ++e) red[(warp * LPR + lane) * 16 + e] = (double)v[e];
            }
          }
          consumers_sync_or(false);
          if (threadIdx.x < LPR) {
            const size_t base = partial_base(cur);
            for (int e = 0; e < NV; ++e) {
              double sum = 0.0;
              for (int w = 0; w < kConsumerWarps; ++w) sum += red[(w * LPR + threadIdx.x) * 16 + e];
              a.partials[base + partial_entry(e)] = sum;
            }
          }
          unwritten = cur + 1;
        }
        if (threadIdx.x < LPR)
          for (int c = unwritten; c < slice; ++c)
            for (int e = 0; e < NV; ++e) a.partials[partial_base(c) + partial_entry(e)] = 0.0;
        unwritten = slice;
      }
      if (slice >= L.n_slices) break;
      cur = slice;
      Z = reinterpret_cast<T*>(a.z) + (size_t)slice * L.D * BS;
      consumers_sync_or(false);  // the previous slice's coefficients have been read
      if (MODE != kModeApply && threadIdx.x < LPR * NVC) {
        const int ln = threadIdx.x / NVC, e = threadIdx.x % NVC;
        const size_t gidx = (size_t)((slice * BS + ln * VW) / DS) * NVG + e;
        s_mz[ln * 16 + e] = (T)a.mz[gidx];
        s_cp[ln * 16 + e] = has_prev ? (T)a.cp[gidx] : (T)0;
      }
      consumers_sync_or(false);
      psum = Pair32{};
#pragma unroll
      for (int e = 0; e < NV; ++e) acc[e] = (T)0;
    }
    if (aborted) continue;

    // (the tile's index: from the table for the uniform terms, whose tiles are short, else
    // with the own tile's stage -- 1% and 5% better so)
    uint32_t ut = UNI ? tt.tile_order[(uint32_t)gt & tile_mask] : 0u;
    const T* sp;
    // own tile: diagonal and in-tile terms
    if (!acquire(sp, 0)) {
      aborted = true;
      continue;
    }
    const T* const own = sp;
    const int n_st = stage[at].what;
    if constexpr (!UNI) ut = stage[at].tile;
    const uint32_t row0 = ut << kTileBits;
    T xo[RPT][VW], y[RPT][VW];
    {
      T dg[RPT];
      tile_diagonal<T, RPT, RG>(dg, s_low, own + kTileBytes / sizeof(T), rg, tt.dg);
      load_rows<kStep>(xo, own + rgoff);
#pragma unroll
      for (int m = 0; m < RPT; ++m)
#pragma unroll
        for (int v = 0; v < VW; ++v) y[m][v] = dg[m] * xo[m][v];
    }
    own_terms<UNI, MODE == kModeApply, RG, kStep>(y, xo, own, rgoff, tt, s_reg, grp, lanet, act_lane, act_grp);
    release();
    // Partner tiles, in the producer's order: opposite-spin pairs, single-spin patterns, the
    // flat ones in use.
    auto single = [&](const PatS<T>& A) {
      single_terms<UNI, MODE == kModeApply, kStep>(y, sp, rgoff, rg, A, (ut & A.high) != 0u, lanet);
    };
    if constexpr (UNI) {
      for (int st = 0; st < n_st;) {
        if (!acquire(sp, 0)) {
          aborted = true;
          break;
        }
        const int p = stage[at].what;
        if (p < nsingle) {
          single(pat[p]);
          release();
          ++st;
          continue;
        }
        const T cA = stage[at].c;
        if (n_st - st > 1) {  // two at a time: their loads overlap
          const T* sb;
          if (!acquire(sb, 1)) {
            aborted = true;
            break;
          }
          rows_fma2<kStep>(y, sp + rgoff, cA, sb + rgoff, stage[at].c);
          release2();
          st += 2;
        } else {
          rows_fma<kStep>(y, sp + rgoff, cA);
          release();
          ++st;
        }
      }
    } else {
      for (int st = 0; st < npair;) {
        if (!acquire(sp, 0)) {
          aborted = true;
          break;
        }
        const int what = stage[at].what;
        const PatS<T>& A = pat[what & (kJoint - 1)];
        if (!(what & kJoint)) {
          single(A);
          release();
          ++st;
          continue;
        }
        // A group whose high spin is down (here) and one whose is up (the next stage), with the
        // same in-tile partners: term l of the first acts on the rows whose spin l is up, of the
        // second on the others, so every row takes exactly one of the two.
        const T* sb;
        if (!acquire(sb, 1)) {
          aborted = true;
          break;
        }
        const PatS<T>& B = pat[stage[at].what];
        pair_terms<kStep>(y, sp, sb, rgoff, rg, A, B, lanet);
        release2();
        st += 2;
      }
      if (aborted) continue;
      for (int p = npair; p < npair + nsingle; ++p) {
        if (!acquire(sp, 0)) {
          aborted = true;
          break;
        }
        single(pat[p]);
        release();
      }
      if (aborted) continue;
      // partner rows are the same rows: one coefficient per tile, from the producer
      int left = n_st - npair - nsingle;
      for (; left > 1; left -= 2) {
        const T* sb;
        if (!acquire(sp, 0)) {
          aborted = true;
          break;
        }
        const T cA = stage[at].c;
        if (!acquire(sb, 1)) {
          aborted = true;
          break;
        }
        rows_fma2<kStep>(y, sp + rgoff, cA, sb + rgoff, stage[at].c);
        release2();
      }
      if (!aborted && left) {
        if (!acquire(sp, 0)) {
          aborted = true;
        } else {
          rows_fma<kStep>(y, sp + rgoff, stage[at].c);
          release();
        }
      }
    }
    if (aborted) continue;
    // Z = (H W) M + W_prev Cp, row by row, with the W_j^T Z partial sums
    const T* Pp = nullptr;
    if (has_prev) {
      if (!acquire(sp, 0)) {
        aborted = true;
        continue;
      }
      Pp = sp;
    }
    T* const zrow = Z + (size_t)row0 * BS + rgoff;  // this thread's first row of the tile
    if constexpr (MODE == kModeApply) {  // Z = H W
#pragma unroll
      for (int m = 0; m < RPT; ++m) VecIO<T, VW>::st_cs(zrow + m * kStep, y[m]);
    } else {
      // this lane's mixing coefficients, read per tile (broadcast shared-memory reads)
      // so they hold no registers while the partner tiles are consumed. M_j is upper
      // triangular (the inverse Cholesky factor, exact zeros below the diagonal), so
      // z = y M_j skips the zero products: the same fma chain, ended early.
      T mz[NVC], cp[NVC];
#pragma unroll
      for (int e = 0; e < NVC; ++e) {
        mz[e] = s_mz[lane * 16 + e];
        cp[e] = s_cp[lane * 16 + e];
      }
      if constexpr (HG) {
        // the row's DS columns: this lane holds columns lane*VW .. lane*VW+VW-1; the whole
        // row of Z is formed (static register indices) and the lane keeps its half
#pragma unroll
        for (int m = 0; m < RPT; ++m) {
          T yf[DS], xf[DS], zf[DS];
#pragma unroll
          for (int v = 0; v < VW; ++v) {
            const T yo = __shfl_xor_sync(0xffffffffu, y[m][v], 1);
            const T xx = __shfl_xor_sync(0xffffffffu, xo[m][v], 1);
            yf[v] = lane == 0 ? y[m][v] : yo;
            yf[VW + v] = lane == 0 ? yo : y[m][v];
            xf[v] = lane == 0 ? xo[m][v] : xx;
            xf[VW + v] = lane == 0 ? xx : xo[m][v];
          }
#pragma unroll
          for (int j = 0; j < DS; ++j) {
            T t = (T)0;
#pragma unroll
            for (int i = 0; i <= j; ++i) t = fma(yf[i], mz[i * DS + j], t);
            zf[j] = t;
          }
          if (has_prev) {
            T xp[VW], pf[DS];
            VecIO<T, VW>::ld_rw(xp, Pp + rgoff + m * kStep);
#pragma unroll
            for (int v = 0; v < VW; ++v) {
              const T po = __shfl_xor_sync(0xffffffffu, xp[v], 1);
              pf[v] = lane == 0 ? xp[v] : po;
              pf[VW + v] = lane == 0 ? po : xp[v];
            }
#pragma unroll
            for (int j = 0; j < DS; ++j) {
              T t = zf[j];
#pragma unroll
              for (int i = 0; i < DS; ++i) t = fma(pf[i], cp[i * DS + j], t);
              zf[j] = t;
            }
          }
          T z[VW];
#pragma unroll
          for (int v = 0; v < VW; ++v) z[v] = lane == 0 ? zf[v] : zf[VW + v];
          VecIO<T, VW>::st_cs(zrow + m * kStep, z);
          if (MODE == kModePass1) {
#pragma unroll
            for (int i = 0; i < DS; ++i)
#pragma unroll
              for (int jj = 0; jj < VW; ++jj) acc[i * VW + jj] = fma(xf[i], z[jj], acc[i * VW + jj]);
          }
        }
      } else
#pragma unroll
      for (int m = 0; m < RPT; ++m) {
        T z[VW];
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int j = 0; j < DS; ++j) {
            T t = (T)0;
#pragma unroll
            for (int i = 0; i <= j; ++i) t = fma(y[m][g * DS + i], mz[g * NVG + i * DS + j], t);
            z[g * DS + j] = t;
          }
        if (has_prev) {
          T xp[VW];
          VecIO<T, VW>::ld_rw(xp, Pp + rgoff + m * kStep);
#pragma unroll
          for (int g = 0; g < NG; ++g)
#pragma unroll
            for (int j = 0; j < DS; ++j) {
              T t = z[g * DS + j];
#pragma unroll
              for (int i = 0; i < DS; ++i) t = fma(xp[g * DS + i], cp[g * NVG + i * DS + j], t);
              z[g * DS + j] = t;
            }
        }
        VecIO<T, VW>::st_cs(zrow + m * kStep, z);
        if (MODE == kModePass1) {
#pragma unroll
          for (int g = 0; g < NG; ++g)
#pragma unroll
            for (int i = 0; i < DS; ++i)
#pragma unroll
              for (int j = 0; j < DS; ++j)
                acc[g * NVG + i * DS + j] = fma(xo[m][g * DS + i], z[g * DS + j], acc[g * NVG + i * DS + j]);
        }
      }
      if (has_prev) release();
      if constexpr (TILE_SUMS) {
        psum.add(warp_sum(acc));
#pragma unroll
        for (int e = 0; e < NV; ++e) acc[e] = (T)0;
      }
    }
  }
  if (aborted && threadIdx.x == 0) atomicOr(a.err, 1u);
}

// ---------------------------------------------------------------- orthogonalisation

// Block (bx, by) of a gx x n_slices grid of the orthogonalisation (grid-stride rows as
// in spmm_block).
//
// float32 rows of two 16-byte lanes (the tiled layout): a thread's products are summed in
// float32 over kOrthChain rows only, then over the warp and the thread's further rows as
// pairs of floats. How many rows a thread takes follows the grid (3 of 2^16 states with 152
// blocks a slice, 85 with 6), and a plain float32 sum over them made B_j's rounding grow with
// the number of bath vectors (N = 19, 1300 vectors: 5e-9 to 6e-8 of B_1).
constexpr int kOrthChain = 16;
template <typename T, int DS, int VW, bool PASS1, bool COH = false>
__device__ __forceinline__ void orth_block(const Layout& L, const T* __restrict__ Wg, T* __restrict__ Zg,
                                           const double* cw, double* partials, T* psi, const double* e,
                                           int nb, int bx, int by, int gx) {
  constexpr int NG = VW / DS;
  constexpr int NVG = DS * DS;
  const int tpr = L.TPR, rpb = kThreads / tpr;
  const int lane = threadIdx.x % tpr, rs = threadIdx.x / tpr;
  const int slice = by;
  const size_t soff = (size_t)slice * L.D * L.Bs + (size_t)lane * VW;
  const T* W = Wg + soff;
  T* Z = Zg + soff;
  const int g0 = (slice * L.Bs + lane * VW) / DS;
  const size_t bstride = (size_t)L.D * L.B;  // elements per psi block
  T c[NG][DS][DS];
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int i = 0; i < DS; ++i)
#pragma unroll
      for (int j = 0; j < DS; ++j) c[g][i][j] = (T)cw[(size_t)(g0 + g) * NVG + i * DS + j];
  T acc[NG][DS][DS];
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int i = 0; i < DS; ++i)
#pragma unroll
      for (int j = 0; j < DS; ++j) acc[g][i][j] = (T)0;
  // pass 2: this slice's E coefficients for all nb betas, as T, in shared memory
  extern __shared__ __align__(16) unsigned char smem_e[];
  T* sE = reinterpret_cast<T*>(smem_e);
  const int gs = L.groups_per_slice();
  if (!PASS1) {
    const int ngs = L.n_groups();
    for (int i = threadIdx.x; i < nb * gs * NVG; i += blockDim.x) {
      const int bi = i / (gs * NVG), rem = i % (gs * NVG);
      sE[i] = (T)e[(size_t)bi * ngs * NVG + (size_t)slice * gs * NVG + rem];
    }
    __syncthreads();
  }
  // (whole blocks of rows: every thread of a warp takes part in the warp's sums)
  const bool chains = PASS1 && sizeof(T) == 4 && tpr == 2 && (L.D & (rpb - 1)) == 0;
  Pair32 psum;  // the warp's sum number warp_sum_index of this lane's column chunk
  int in_chain = 0;
  auto fold = [&]() {
    if constexpr (PASS1 && sizeof(T) == 4) {
      Pair32 v[NG * NVG];
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int i = 0; i < DS; ++i)
#pragma unroll
          for (int j = 0; j < DS; ++j) v[g * NVG + i * DS + j].hi = j >= i ? acc[g][i][j] : acc[g][j][i];
      psum.add(warp_sum(v));
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int i = 0; i < DS; ++i)
#pragma unroll
          for (int j = 0; j < DS; ++j) acc[g][i][j] = (T)0;
      in_chain = 0;
    }
  };
  for (int64_t s = (int64_t)bx * rpb + rs; s < L.D; s += (int64_t)gx * rpb) {
    T x[VW], z[VW];
    ld_vec<T, VW, COH>(x, W + (size_t)s * L.Bs);
    VecIO<T, VW>::ld_rw(z, Z + (size_t)s * L.Bs);
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int j = 0; j < DS; ++j) {
        T t = z[g * DS + j];
#pragma unroll
        for (int i = 0; i < DS; ++i) t = fma(x[g * DS + i], c[g][i][j], t);
        z[g * DS + j] = t;
      }
    VecIO<T, VW>::st(Z + (size_t)s * L.Bs, z);
    if (PASS1) {
      // the upper triangle: the lower one is the same products (float64 is bound by its
      // pipe: N = 19, d_s = 4, 8 vectors 0.274 -> 0.234 ms)
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int i = 0; i < DS; ++i)
#pragma unroll
          for (int j = i; j < DS; ++j) acc[g][i][j] = fma(z[g * DS + i], z[g * DS + j], acc[g][i][j]);
      if (chains && ++in_chain == kOrthChain) fold();
    } else {
      for (int bi = 0; bi < nb; ++bi) {
        T* P = psi + bi * bstride + soff + (size_t)s * L.Bs;
        T p[VW];
        VecIO<T, VW>::ld_rw(p, P);
        const T* eb = sE + ((size_t)bi * gs + (size_t)lane * NG) * NVG;
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int j = 0; j < DS; ++j) {
            T t = p[g * DS + j];
#pragma unroll
            for (int i = 0; i < DS; ++i) t = fma(z[g * DS + i], eb[g * NVG + i * DS + j], t);
            p[g * DS + j] = t;
          }
        VecIO<T, VW>::st(P, p);
      }
    }
  }
  if (PASS1) {
    if constexpr (sizeof(T) == 4)
      if (chains) {
        if (in_chain) fold();
        warp_sums_store<NG * NVG>(psum, partials, (size_t)by * gx + bx);
        return;
      }
    T vals[NG * NVG];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < DS; ++i)
#pragma unroll
        for (int j = 0; j < DS; ++j) vals[g * NVG + i * DS + j] = j >= i ? acc[g][i][j] : acc[g][j][i];
    block_reduce_store<NG, NVG, T>(vals, tpr, partials, L.groups_per_slice(), (size_t)by * gx + bx);
  }
}

template <typename T, int DS, int VW, bool PASS1>
__global__ void __launch_bounds__(kThreads) k_orth(Layout L, const T* __restrict__ Wg,
                                                   T* __restrict__ Zg, const double* cw,
                                                   double* partials, T* psi, const double* e,
                                                   int nb) {
  orth_block<T, DS, VW, PASS1>(L, Wg, Zg, cw, partials, psi, e, nb, blockIdx.x, blockIdx.y, gridDim.x);
}

// psi_beta = W_1 E_{1,beta} (start of pass 2).
template <typename T, int DS, int VW>
__global__ void __launch_bounds__(kThreads) k_psi_init(Layout L, const T* __restrict__ Wg,
                                                       T* psi, const double* e, int nb) {
  constexpr int NG = VW / DS;
  constexpr int NVG = DS * DS;
  const int tpr = L.TPR, rpb = kThreads / tpr;
  const int lane = threadIdx.x % tpr, rs = threadIdx.x / tpr;
  const int slice = blockIdx.y;
  const size_t soff = (size_t)slice * L.D * L.Bs + (size_t)lane * VW;
  const int g0 = (slice * L.Bs + lane * VW) / DS;
  const size_t bstride = (size_t)L.D * L.B;
  const int ngs = L.n_groups();
  for (int64_t s = (int64_t)blockIdx.x * rpb + rs; s < L.D; s += (int64_t)gridDim.x * rpb) {
    T x[VW];
    VecIO<T, VW>::ld(x, Wg + soff + (size_t)s * L.Bs);
    for (int bi = 0; bi < nb; ++bi) {
      const double* eb = e + (size_t)bi * ngs * NVG;
      T p[VW];
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int j = 0; j < DS; ++j) {
          T t = (T)0;
#pragma unroll
          for (int i = 0; i < DS; ++i) t = fma(x[g * DS + i], (T)eb[(size_t)(g0 + g) * NVG + i * DS + j], t);
          p[g * DS + j] = t;
        }
      VecIO<T, VW>::st(psi + bi * bstride + soff + (size_t)s * L.Bs, p);
    }
  }
}

// psi_beta += sum_{a < m} W_a E_{j0+a,beta} (pass 2, m kept basis blocks): each psi
// element is read and written once for m steps instead of once per step.
template <typename T, int DS, int VW>
__global__ void __launch_bounds__(kThreads) k_psi_batch(Layout L, PsiBatch wb, int m, T* psi,
                                                        const double* e, size_t estride, int nb) {
  constexpr int NG = VW / DS;
  constexpr int NVG = DS * DS;
  const int tpr = L.TPR, rpb = kThreads / tpr;
  const int lane = threadIdx.x % tpr, rs = threadIdx.x / tpr;
  const int slice = blockIdx.y;
  const size_t soff = (size_t)slice * L.D * L.Bs + (size_t)lane * VW;
  const size_t bstride = (size_t)L.D * L.B;
  const int gs = L.groups_per_slice(), ngs = L.n_groups();
  // this slice's E coefficients, [a][beta][group][DS*DS], as T
  extern __shared__ __align__(16) unsigned char smem_e[];
  T* sE = reinterpret_cast<T*>(smem_e);
  const int per = nb * gs * NVG;
  for (int i = threadIdx.x; i < m * per; i += blockDim.x) {
    const int a = i / per, rem = i % per, bi = rem / (gs * NVG), r2 = rem % (gs * NVG);
    sE[i] = (T)e[(size_t)a * estride + (size_t)bi * ngs * NVG + (size_t)slice * gs * NVG + r2];
  }
  __syncthreads();
  for (int64_t s = (int64_t)blockIdx.x * rpb + rs; s < L.D; s += (int64_t)gridDim.x * rpb) {
    T x[kPsiBatchMax][VW];
#pragma unroll
    for (int a = 0; a < kPsiBatchMax; ++a)
      if (a < m) VecIO<T, VW>::ld(x[a], reinterpret_cast<const T*>(wb.w[a]) + soff + (size_t)s * L.Bs);
    for (int bi = 0; bi < nb; ++bi) {
      T* P = psi + bi * bstride + soff + (size_t)s * L.Bs;
      T p[VW];
      VecIO<T, VW>::ld_rw(p, P);
#pragma unroll
      for (int a = 0; a < kPsiBatchMax; ++a) {
        if (a >= m) break;
        const T* eb = sE + ((size_t)(a * nb + bi) * gs + (size_t)lane * NG) * NVG;
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int j = 0; j < DS; ++j) {
            T t = p[g * DS + j];
#pragma unroll
            for (int i = 0; i < DS; ++i) t = fma(x[a][g * DS + i], eb[g * NVG + i * DS + j], t);
            p[g * DS + j] = t;
          }
      }
      VecIO<T, VW>::st(P, p);
    }
  }
}

// Gram partials of one psi block. The Gram is accumulated in float64 whatever the
// vectors' precision (eq. rho_est): a product of two float32 values is exact in float64,
// so each fma rounds only the sum. Only the upper triangle is summed; the lower one is
// its mirror (the same products, so the same bits).
template <typename T, int DS, int VW>
__global__ void __launch_bounds__(kThreads) k_final_gram(Layout L, const T* __restrict__ P,
                                                         double* partials) {
  constexpr int NG = VW / DS;
  constexpr int NVG = DS * DS;
  const int tpr = L.TPR, rpb = kThreads / tpr;
  const int lane = threadIdx.x % tpr, rs = threadIdx.x / tpr;
  const int slice = blockIdx.y;
  const size_t soff = (size_t)slice * L.D * L.Bs + (size_t)lane * VW;
  double acc[NG][DS][DS];
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int i = 0; i < DS; ++i)
#pragma unroll
      for (int j = 0; j < DS; ++j) acc[g][i][j] = 0.0;
  for (int64_t s = (int64_t)blockIdx.x * rpb + rs; s < L.D; s += (int64_t)gridDim.x * rpb) {
    T p[VW];
    VecIO<T, VW>::ld(p, P + soff + (size_t)s * L.Bs);
    double pd[VW];
#pragma unroll
    for (int v = 0; v < VW; ++v) pd[v] = (double)p[v];
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < DS; ++i)
#pragma unroll
        for (int j = i; j < DS; ++j) acc[g][i][j] = fma(pd[g * DS + i], pd[g * DS + j], acc[g][i][j]);
  }
  double vals[NG * NVG];
#pragma unroll
  for (int g = 0; g < NG; ++g)
#pragma unroll
    for (int i = 0; i < DS; ++i)
#pragma unroll
      for (int j = 0; j < DS; ++j) vals[g * NVG + i * DS + j] = j >= i ? acc[g][i][j] : acc[g][j][i];
  block_reduce_store<NG, NVG, double>(vals, tpr, partials, L.groups_per_slice(),
                                       (size_t)blockIdx.y * gridDim.x + blockIdx.x);
}

// Stored-basis Gram for float64 blocks and for float32 rows other than 32 bytes (blocks of
// fewer than 2^kTileBits states; k_gram_rows takes the rest): psi_beta = sum_{j=1..k} W_j E_{j,beta} row by row (the same
// fma sequence as the two-pass accumulation, so the result is bit-identical) and
// the partial sums of psi_beta^T psi_beta, for up to kGramBetas betas per launch.
// W_j = W1 + (j-1) * D * B elements; e: [j][beta (stride nbs)][group][DS*DS].
constexpr int kGramBetas = 4;

template <typename T, int DS>
struct RowVec;  // DS consecutive coefficients as one shared-memory load
template <>
struct RowVec<float, 4> {
  __device__ static void ld(float* r, const float* p) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    r[0] = v.x; r[1] = v.y; r[2] = v.z; r[3] = v.w;
  }
};
template <>
struct RowVec<float, 2> {
  __device__ static void ld(float* r, const float* p) {
    const float2 v = *reinterpret_cast<const float2*>(p);
    r[0] = v.x; r[1] = v.y;
  }
};
template <>
struct RowVec<float, 1> {
  __device__ static void ld(float* r, const float* p) { r[0] = *p; }
};
template <>
struct RowVec<double, 4> {
  __device__ static void ld(double* r, const double* p) {
    const double2 a = *reinterpret_cast<const double2*>(p);
    const double2 b = *reinterpret_cast<const double2*>(p + 2);
    r[0] = a.x; r[1] = a.y; r[2] = b.x; r[3] = b.y;
  }
};
template <>
struct RowVec<double, 2> {
  __device__ static void ld(double* r, const double* p) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    r[0] = v.x; r[1] = v.y;
  }
};
template <>
struct RowVec<double, 1> {
  __device__ static void ld(double* r, const double* p) { r[0] = *p; }
};

// Each thread takes two rows at a time so every coefficient row read from shared
// memory serves both.
template <typename T, int DS, int VW, int NBT>
__global__ void __launch_bounds__(kThreads) k_gram_stored(Layout L, const T* __restrict__ W1, int k,
                                                          const double* e, int nbs, int b0, int nb,
                                                          double* partials, size_t pstride) {
  constexpr int NG = VW / DS;
  constexpr int NVG = DS * DS;
  extern __shared__ __align__(16) unsigned char smem_g[];
  T* sE = reinterpret_cast<T*>(smem_g);  // [j][bi][gs][NVG]
  const int tpr = L.TPR, rpb = kThreads / tpr;
  const int lane = threadIdx.x % tpr, rs = threadIdx.x / tpr;
  const int slice = blockIdx.y;
  const int gs = L.groups_per_slice(), ng = L.n_groups();
  const size_t soff = (size_t)slice * L.D * L.Bs + (size_t)lane * VW;
  const size_t bstride = (size_t)L.D * L.B;
  for (int i = threadIdx.x; i < k * nb * gs * NVG; i += blockDim.x) {
    const int j = i / (nb * gs * NVG);
    const int rem = i % (nb * gs * NVG);
    const int bi = rem / (gs * NVG), r2 = rem % (gs * NVG);
    sE[i] = (T)e[(((size_t)j * nbs + b0 + bi) * ng) * NVG + (size_t)slice * gs * NVG + r2];
  }
  __syncthreads();
  // the Gram in float64 (upper triangle; see k_final_gram)
  double acc[NBT][NG][DS][DS];
#pragma unroll
  for (int bi = 0; bi < NBT; ++bi)
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < DS; ++i)
#pragma unroll
        for (int j = 0; j < DS; ++j) acc[bi][g][i][j] = 0.0;
  // Rows s and s + stride form a pair; the accumulation order per row is the same
  // as for single rows (rows are visited in the same sequence per thread).
  const int64_t stride = (int64_t)gridDim.x * rpb;
  for (int64_t s0 = (int64_t)blockIdx.x * rpb + rs; s0 < L.D; s0 += 2 * stride) {
    const int64_t s1 = s0 + stride;
    const bool two = s1 < L.D;
    T psi[2][NBT][VW];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int bi = 0; bi < NBT; ++bi)
#pragma unroll
        for (int v = 0; v < VW; ++v) psi[h][bi][v] = (T)0;
    auto step = [&](int j, const T (&x)[2][VW]) {
#pragma unroll
      for (int bi = 0; bi < NBT; ++bi) {
        if (bi >= nb) break;
        const T* eb = sE + (((size_t)j * nb + bi) * gs + (size_t)lane * NG) * NVG;
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int i = 0; i < DS; ++i) {
            T er[DS];
            RowVec<T, DS>::ld(er, eb + g * NVG + i * DS);
#pragma unroll
            for (int jj = 0; jj < DS; ++jj) {
              psi[0][bi][g * DS + jj] = fma(x[0][g * DS + i], er[jj], psi[0][bi][g * DS + jj]);
              psi[1][bi][g * DS + jj] = fma(x[1][g * DS + i], er[jj], psi[1][bi][g * DS + jj]);
            }
          }
      }
    };
    int j = 0;
    for (; j + 4 <= k; j += 4) {  // four blocks' loads in flight before their use
      T x[4][2][VW];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const T* wj = W1 + (size_t)(j + u) * bstride + soff;
        VecIO<T, VW>::ld(x[u][0], wj + (size_t)s0 * L.Bs);
        if (two) VecIO<T, VW>::ld(x[u][1], wj + (size_t)s1 * L.Bs);
        else
#pragma unroll
          for (int v = 0; v < VW; ++v) x[u][1][v] = (T)0;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) step(j + u, x[u]);
    }
    for (; j < k; ++j) {
      T x[2][VW];
      const T* wj = W1 + (size_t)j * bstride + soff;
      VecIO<T, VW>::ld(x[0], wj + (size_t)s0 * L.Bs);
      if (two) VecIO<T, VW>::ld(x[1], wj + (size_t)s1 * L.Bs);
      else
#pragma unroll
        for (int v = 0; v < VW; ++v) x[1][v] = (T)0;
      step(j, x);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (h == 1 && !two) break;
#pragma unroll
      for (int bi = 0; bi < NBT; ++bi) {
        double pd[VW];
#pragma unroll
        for (int v = 0; v < VW; ++v) pd[v] = (double)psi[h][bi][v];
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int i = 0; i < DS; ++i)
#pragma unroll
            for (int j = i; j < DS; ++j)
              acc[bi][g][i][j] = fma(pd[g * DS + i], pd[g * DS + j], acc[bi][g][i][j]);
      }
    }
  }
#pragma unroll
  for (int bi = 0; bi < NBT; ++bi) {  // static indices keep acc in registers
    if (bi < nb) {
      double vals[NG * NVG];
#pragma unroll
      for (int g = 0; g < NG; ++g)
#pragma unroll
        for (int i = 0; i < DS; ++i)
#pragma unroll
          for (int j = 0; j < DS; ++j)
            vals[g * NVG + i * DS + j] = j >= i ? acc[bi][g][i][j] : acc[bi][g][j][i];
      block_reduce_store<NG, NVG, double>(vals, tpr, partials + (size_t)bi * pstride, gs,
                                           (size_t)blockIdx.y * gridDim.x + blockIdx.x);
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------- float32 Gram on 32-byte rows
//
// The Gram form's kernel for float32 blocks with 32-byte rows (the tiled layout), all betas
// in one launch: psi_beta = sum_{j <= k_beta} W_j E_{j,beta} row by row (per element the fma
// sequence of the other kernels, j then i ascending) and the sums of psi_beta^T psi_beta in
// float64 (k_final_gram).
//
// What bounds it. GB300 issues 1.8 float64 fmas and 2.1 float32 -> float64 conversions per
// clock and SM against 128 float32 fmas (measured), and a d_s = 4 row costs 10 products and
// 4 conversions per beta: k_gram_stored, which this kernel replaces here, spent its time on
// that pipe (63% busy under ncu) with 2 warps a scheduler, beside which nothing else ran.
// So the conversions are integer operations (to_double), the basis rows come through
// per-thread copy rings, and small blocks without barriers let one warp's float64 products
// run beside the others' float32 fmas. Register prefetch instead of the rings stalled on
// loads at every part (long_scoreboard 46%); a ring shared by a block kept its warps in step.
//
// A group of up to NBT betas shares one reading of the basis; the groups of one row range
// are neighbours in the grid and take betas of the same spread of k_beta (every nz-th of the
// betas in order of k_beta), so they move through the rows together and all but the first
// find them in L2. At step j only the group's betas with k_beta > j are updated.
//
// Per solve, before and after: ladder N = 20 (n_v = 50, 16 betas, 30 steps) 50.0 -> 24.4 ms;
// long-range XY N = 16 (n_v = 400, 8 betas) 34.6 -> 9.0 ms; long-range XXZ N = 22 (d_s = 2,
// n_v = 16, 32 betas, 40 steps) 47.0 -> 23.4 ms; 48 small solves 87.7 -> 13.7 ms; one beta at
// N = 22 (HBM, 6.8 TB/s) 10.4 ms as before.
constexpr int kGramThreads = 128;
constexpr int kGramStages = 8;  // steps in flight per thread (12: 4% slower)
constexpr int kGramChunk = 512;  // rows per block and pass, whatever R: the sums' order
struct GramBetas {
  uint16_t k[kGramLaunchBetas];     // basis blocks each beta needs, descending
  uint8_t beta[kGramLaunchBetas];   // and its place in the launch's betas
};

// (double)x with integer operations, of 2^64 x so that subnormals (a bath vector whose lowest
// Ritz value lies so far above E0 that exp(-beta (t - E0) / 2) leaves float32's normal range)
// need no branch: the exponent rebiased by 896 - 64 and the mantissa moved up; infinities and
// NaN keep their exponent of ones. (|psi| stays of the order of 1: far below 2^64. Converting
// the subnormals on their own took the ladder's Gram from 24.4 to 26 ms.)
__device__ __forceinline__ double to_double(float x) {
  const uint32_t u = __float_as_uint(x * 0x1p64f), a = u & 0x7fffffffu;
  uint32_t hi = (a >> 3) + 0x34000000u;
  if (a >= 0x7f800000u) hi += 0x3c000000u;
  if (a == 0u) hi = 0u;
  return __hiloint2double((int)(hi | (u & 0x80000000u)), (int)(u << 29));
}

// NBT: the largest group. FINAL: W1 holds nb blocks psi_beta (group size 1).
template <int DS, int NBT, bool FINAL>
__global__ void __launch_bounds__(kGramThreads, 3)
    k_gram_rows(Layout L, const float* __restrict__ W1, GramBetas gb, const double* e, int nbs, int b0, int nb,
                int nz, double* partials, size_t pstride) {
  constexpr int VW = 4, NG = VW / DS, NVG = DS * DS;
  constexpr int R = NBT >= 4 ? 2 : 4;   // rows per thread at a time (psi in registers)
  constexpr int RS = kGramThreads / 2;  // rows between them
  constexpr int CO = VW * DS;           // coefficients per lane, step and beta
  extern __shared__ __align__(16) unsigned char smem_g[];
  float* const sE = reinterpret_cast<float*>(smem_g);  // [j][bi][lane][CO]
  __shared__ double red[kGramThreads / 32][2][NG * NVG];
  const int z = blockIdx.x % nz, bx = blockIdx.x / nz, gx = L.gridx;
  const int slice = blockIdx.y, gs = 2 * NG, ng = L.n_groups();
  const int lane = threadIdx.x & 1, rs = threadIdx.x >> 1;
  const size_t bstride = (size_t)L.D * L.B;
  const float* const base =  // this thread's 16 bytes of row 0
      W1 + (size_t)slice * L.D * 8 + (FINAL ? (size_t)z * bstride : 0) + (size_t)rs * 8 + lane * VW;
  int kb[NBT];  // steps of the group's betas, descending (0: none)
#pragma unroll
  for (int bi = 0; bi < NBT; ++bi) kb[bi] = bi * nz + z < nb ? (FINAL ? 1 : (int)gb.k[bi * nz + z]) : 0;
  const int kz = kb[0];
  if (!FINAL) {
    for (int i = threadIdx.x; i < kz * NBT * 2 * CO; i += kGramThreads) {
      const int r = i % (2 * CO), bi = i / (2 * CO) % NBT, j = i / (2 * CO * NBT);
      const int q = bi * nz + z;
      if (q < nb && j < (int)gb.k[q])
        sE[i] = (float)e[((size_t)j * nbs + b0 + gb.beta[q]) * ng * NVG + (size_t)slice * gs * NVG + r];
    }
    __syncthreads();
  }
  double acc[NBT][NG][DS][DS];
#pragma unroll
  for (int bi = 0; bi < NBT; ++bi)
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < DS; ++i)
#pragma unroll
        for (int j = 0; j < DS; ++j) acc[bi][g][i][j] = 0.0;
  // Each thread copies its own 16 bytes of R rows per step into its own places of a ring of
  // kGramStages steps (cp.async: no barrier, the warps drift apart freely), across the
  // boundaries of row parts, so the next part's first steps arrive under this part's sums.
  float* const ring = sE + (FINAL ? 0 : (size_t)kz * NBT * 2 * CO) + threadIdx.x * VW;
  constexpr int kStage = R * kGramThreads * VW;  // floats
  const int64_t chunks = L.D / kGramChunk;
  const int64_t parts = (chunks - bx + gx - 1) / gx * (kGramChunk / (R * RS));  // of this block
  int64_t lp = 0;  // the part and step of the next copy
  int lj = 0, lslot = 0;
  const float* src = base + (size_t)bx * kGramChunk * 8;
  auto issue = [&]() {
    if (lp < parts) {
      const float* q = src + (size_t)lj * bstride;
      float* d = ring + lslot * kStage;
#pragma unroll
      for (int r = 0; r < R; ++r)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_u32(d + r * kGramThreads * VW)),
                     "l"(q + (size_t)r * RS * 8)
                     : "memory");
      if (++lj == kz) {
        lj = 0;
        ++lp;
        src += (size_t)R * RS * 8;
        if (lp % (kGramChunk / (R * RS)) == 0) src += (size_t)(gx - 1) * kGramChunk * 8;
      }
    }
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    if (++lslot == kGramStages) lslot = 0;
  };
#pragma unroll
  for (int u = 0; u < kGramStages - 1; ++u) issue();
  int slot = 0;
  for (int64_t part = 0; part < parts; ++part) {
    float psi[R][NBT][VW];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int bi = 0; bi < NBT; ++bi)
#pragma unroll
        for (int v = 0; v < VW; ++v) psi[r][bi][v] = 0.0f;
    for (int j = 0; j < kz; ++j) {
      issue();  // into the place freed one step ago
      asm volatile("cp.async.wait_group %0;\n" ::"n"(kGramStages - 1) : "memory");
      float x[R][VW];
#pragma unroll
      for (int r = 0; r < R; ++r) VecIO<float, VW>::ld_rw(x[r], ring + slot * kStage + r * kGramThreads * VW);
      if (++slot == kGramStages) slot = 0;
      if constexpr (FINAL) {
#pragma unroll
        for (int r = 0; r < R; ++r)
#pragma unroll
          for (int v = 0; v < VW; ++v) psi[r][0][v] = x[r][v];
      } else {
#pragma unroll
        for (int bi = 0; bi < NBT; ++bi) {
          if (j >= kb[bi]) break;
          const float* eb = sE + ((size_t)(j * NBT + bi) * 2 + lane) * CO;
#pragma unroll
          for (int g = 0; g < NG; ++g)
#pragma unroll
            for (int i = 0; i < DS; ++i) {
              float er[DS];
              RowVec<float, DS>::ld(er, eb + g * NVG + i * DS);
#pragma unroll
              for (int jj = 0; jj < DS; ++jj)
#pragma unroll
                for (int r = 0; r < R; ++r)
                  psi[r][bi][g * DS + jj] = fmaf(x[r][g * DS + i], er[jj], psi[r][bi][g * DS + jj]);
            }
        }
      }
    }
#pragma unroll
    for (int bi = 0; bi < NBT; ++bi) {
      if (kb[bi] == 0) break;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        double pd[VW];
#pragma unroll
        for (int v = 0; v < VW; ++v) pd[v] = to_double(psi[r][bi][v]);
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int i = 0; i < DS; ++i)
#pragma unroll
            for (int j = i; j < DS; ++j)
              acc[bi][g][i][j] = fma(pd[g * DS + i], pd[g * DS + j], acc[bi][g][i][j]);
      }
    }
  }
  asm volatile("cp.async.wait_all;\n" ::: "memory");
  const int wl = threadIdx.x & 31;
#pragma unroll
  for (int bi = 0; bi < NBT; ++bi) {
    if (kb[bi] == 0) break;
#pragma unroll
    for (int g = 0; g < NG; ++g)
#pragma unroll
      for (int i = 0; i < DS; ++i)
#pragma unroll
        for (int j = i; j < DS; ++j) {
          double x = acc[bi][g][i][j];
#pragma unroll
          for (int o = 2; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
          if (wl < 2) {
            red[threadIdx.x >> 5][wl][g * NVG + i * DS + j] = x;
            red[threadIdx.x >> 5][wl][g * NVG + j * DS + i] = x;
          }
        }
    __syncthreads();
    if (threadIdx.x < 2 * NG * NVG) {
      const int ln = threadIdx.x / (NG * NVG), v = threadIdx.x % (NG * NVG);
      double sum = 0.0;
      for (int w = 0; w < kGramThreads / 32; ++w) sum += red[w][ln][v];
      const int beta = FINAL ? z : (int)gb.beta[bi * nz + z];
      partials[(size_t)beta * pstride + (((size_t)slice * gx + bx) * gs + (size_t)ln * NG) * NVG + v] = sum;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- per-group small steps

constexpr int kSmallThreads = 128;

// Sums the NV partials of group l over the gridx blocks (fixed order: thread t < 128
// takes bx = t, t + 128, ..., then a tree over the 128 sums). Every thread of the block
// must call it; threads beyond the first kSmallThreads only pass the barriers.
template <int NV>
__device__ void reduce_group(const Layout& L, const double* partials, double* out, int l) {
  __shared__ double sh[kSmallThreads];
  const int gs = L.groups_per_slice();
  const int slice = l / gs, gis = l % gs;
  const bool part = threadIdx.x < kSmallThreads;
  for (int v = 0; v < NV; ++v) {
    if (part) {
      double s = 0.0;
      for (int bx = threadIdx.x; bx < L.gridx; bx += kSmallThreads)
        s += partials[((size_t)(slice * L.gridx + bx) * gs + gis) * NV + v];
      sh[threadIdx.x] = s;
    }
    __syncthreads();
    for (int w = kSmallThreads / 2; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[v] = sh[0];
    __syncthreads();
  }
}

template <int DS>
__global__ void k_coef_init(int n_groups, double* mz, double* cp) {
  const int l = blockIdx.x * blockDim.x + threadIdx.x;
  if (l >= n_groups) return;
  for (int i = 0; i < DS; ++i)
    for (int j = 0; j < DS; ++j) {
      mz[(size_t)l * DS * DS + i * DS + j] = i == j ? 1.0 : 0.0;
      cp[(size_t)l * DS * DS + i * DS + j] = 0.0;
    }
}

// After the SpMM, for group l (every thread of the block calls it): A_j and Cw_j.
template <int DS>
__device__ void small_a_group(const Layout& L, const double* partials, const double* mz, double* a_out,
                              double* cw_out, uint32_t* flags, int l) {
  constexpr int NV = DS * DS;
  __shared__ double tot[NV];
  reduce_group<NV>(L, partials, tot, l);
  if (threadIdx.x != 0) return;
  const double* M = mz + (size_t)l * NV;
  double p1[DS][DS], A[DS][DS];
  // P1 = M^T (W^T Z) = Q_j^T Z
  for (int i = 0; i < DS; ++i)
    for (int j = 0; j < DS; ++j) {
      double s = 0.0;
      for (int c = 0; c < DS; ++c) s += M[c * DS + i] * tot[c * DS + j];
      p1[i][j] = s;
    }
  bool finite = true;
  for (int i = 0; i < DS; ++i)
    for (int j = 0; j < DS; ++j) {
      A[i][j] = 0.5 * (p1[i][j] + p1[j][i]);
      finite = finite && isfinite(A[i][j]);
    }
  for (int i = 0; i < DS; ++i)
    for (int j = 0; j < DS; ++j) {
      a_out[(size_t)l * NV + i * DS + j] = A[i][j];
      double s = 0.0;
      for (int c = 0; c < DS; ++c) s += M[i * DS + c] * A[c][j];
      cw_out[(size_t)l * NV + i * DS + j] = -s;
    }
  if (!finite) atomicOr(flags, kFlagNonFinite);
}

template <int DS>
__global__ void k_small_a(Layout L, const double* partials, const double* mz, double* a_out,
                          double* cw_out, uint32_t* flags) {
  small_a_group<DS>(L, partials, mz, a_out, cw_out, flags, blockIdx.x);
}

// One group's Cholesky QR with deflation from the Gram `tot`: B_j, M_{j+1}, Cp_{j+1} = -M_j
// B_j^T. Returns whether a column was dropped.
template <int DS>
__device__ bool qr_group(const double* tot, const double* Mj, double thr_abs_sq, double thr_rel_sq, double* b_out,
                         double* mz_next, double* cp_next, bool& finite) {
  double G[DS][DS], R[DS][DS], Ri[DS][DS];
  bool kept[DS];
  for (int i = 0; i < DS; ++i)
    for (int j = 0; j < DS; ++j) {
      G[i][j] = 0.5 * (tot[i * DS + j] + tot[j * DS + i]);
      R[i][j] = 0.0;
      Ri[i][j] = 0.0;
    }
  // Cholesky G = R^T R column by column, dropping numerically dependent columns
  // (Gram-Schmidt in the G inner product; same rule as a column-wise QR).
  bool dropped = false;
  finite = true;
  for (int c = 0; c < DS; ++c) {
    for (int k = 0; k < c; ++k) {
      if (!kept[k]) continue;
      double s = G[k][c];
      for (int i = 0; i < k; ++i)
        if (kept[i]) s -= R[i][k] * R[i][c];
      R[k][c] = s / R[k][k];
    }
    double piv = G[c][c];
    for (int k = 0; k < c; ++k)
      if (kept[k]) piv -= R[k][c] * R[k][c];
    finite = finite && isfinite(piv);
    if (!(piv > thr_abs_sq) || !(piv > thr_rel_sq * G[c][c])) {
      kept[c] = false;
      R[c][c] = 0.0;
      dropped = true;
    } else {
      kept[c] = true;
      R[c][c] = sqrt(piv);
    }
  }
  // Inverse of R restricted to the kept columns (back substitution), zero elsewhere.
  for (int c = 0; c < DS; ++c) {
    if (!kept[c]) continue;
    Ri[c][c] = 1.0 / R[c][c];
    for (int r = c - 1; r >= 0; --r) {
      if (!kept[r]) continue;
      double s = 0.0;
      for (int m = r + 1; m <= c; ++m)
        if (kept[m]) s += R[r][m] * Ri[m][c];
      Ri[r][c] = -s / R[r][r];
    }
  }
  for (int i = 0; i < DS; ++i)
    for (int j = 0; j < DS; ++j) {
      b_out[i * DS + j] = R[i][j];
      mz_next[i * DS + j] = Ri[i][j];
      double s = 0.0;
      for (int c = 0; c < DS; ++c) s += Mj[i * DS + c] * R[j][c];
      cp_next[i * DS + j] = -s;
    }
  return dropped;
}

// After the orthogonalisation, for group l (every thread of the block calls it): the
// Cholesky QR with deflation -> B_j, M_{j+1}, Cp_{j+1}.
template <int DS>
__device__ void small_b_group(const Layout& L, const double* partials, const double* mz_j, double* b_out,
                              double* mz_next, double* cp_next, double thr_abs_sq, double thr_rel_sq,
                              int n_real, uint32_t* flags, int l) {
  constexpr int NV = DS * DS;
  __shared__ double tot[NV];
  reduce_group<NV>(L, partials, tot, l);
  if (threadIdx.x != 0) return;
  const size_t o = (size_t)l * NV;
  bool finite;
  const bool dropped = qr_group<DS>(tot, mz_j + o, thr_abs_sq, thr_rel_sq, b_out + o, mz_next + o, cp_next + o, finite);
  if (dropped && l < n_real) atomicOr(flags, (uint32_t)RDM_FLAG_DEFLATED);
  if (!finite) atomicOr(flags, kFlagNonFinite);
}

template <int DS>
__global__ void k_small_b(Layout L, const double* partials, const double* mz_j, double* b_out,
                          double* mz_next, double* cp_next, double thr_abs_sq, double thr_rel_sq,
                          int n_real, uint32_t* flags) {
  small_b_group<DS>(L, partials, mz_j, b_out, mz_next, cp_next, thr_abs_sq, thr_rel_sq, n_real, flags,
                    blockIdx.x);
}

// Group blockIdx.x of beta blockIdx.y.
template <int DS>
__global__ void k_reduce_gram(Layout L, const double* partials, size_t pstride, double* gram) {
  constexpr int NV = DS * DS;
  __shared__ double tot[NV];
  reduce_group<NV>(L, partials + blockIdx.y * pstride, tot, blockIdx.x);
  if (threadIdx.x != 0) return;
  for (int v = 0; v < NV; ++v) gram[((size_t)blockIdx.y * L.n_groups() + blockIdx.x) * NV + v] = tot[v];
}

// ---------------------------------------------------------------- packed first pass
//
// The first pass (Algorithm 1's k steps) of several estimates in ONE cooperative
// launch: every block of a persistent grid walks the work units of a phase, and a grid
// barrier separates the phases of a step: SpMM (+ W_j^T Z partials), A_j per bath
// vector, orthogonalisation (+ Gram partials), Cholesky QR per bath vector. A unit is
// exactly one block of the corresponding plain launch of that estimate (block (bx, by)
// of its gridx x n_slices grid, or group l), so each estimate's arithmetic and
// reduction order depend on its own layout only: results are the same whichever
// estimates share the launch and however the units are spread over the grid. Items are
// sorted by k, largest first, so the items still running at step j are a prefix.

// Grid barrier: arrival counter, generation word, error word (zero before the launch).
// The last block to arrive resets the counter and advances the generation; the others
// wait for that with a bounded spin. A wait that gives up sets the error word, and a
// block that sees the error word set leaves at its next barrier.
__device__ __forceinline__ uint32_t ld_acquire_gpu(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ bool grid_barrier(uint32_t* bar, uint32_t& gen) {
  __shared__ int ok_s;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    if (ld_acquire_gpu(bar + 2) != 0u) {
      ok = 0;
    } else if (atomicAdd(bar, 1u) == gridDim.x - 1u) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicExch(bar + 1, gen + 1u);
    } else {
      uint32_t it = 0;
      while (ld_acquire_gpu(bar + 1) == gen) {
        if (++it > (1u << 24) || ld_acquire_gpu(bar + 2) != 0u) {
          atomicOr(bar + 2, 1u);
          ok = 0;
          break;
        }
        if (it > 64) __nanosleep(64);
      }
    }
    __threadfence();
    ok_s = ok;
  }
  __syncthreads();
  ++gen;
  return ok_s != 0;
}

// Unit u of a phase -> its item (largest i with pre[i] <= u among the first n).
__device__ __forceinline__ int packed_item_of(const int* pre, int n, int u) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (pre[mid] <= u)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

template <typename T, int DS, int VW>
__global__ void __launch_bounds__(kThreads) k_pass1_packed(PackedPlan pp) {
  constexpr int NVG = DS * DS;
  uint32_t gen = 0;
  for (int j = 1; j <= pp.k_max; ++j) {
    const int na = pp.active[j];
    // phase A: Z = (H W_j) M_j + W_{j-1} Cp_j and the partial sums of W_j^T Z
    for (int u = blockIdx.x; u < pp.pre_rows[na]; u += gridDim.x) {
      const int i = packed_item_of(pp.pre_rows, na, u);
      const PackedItem& it = pp.items[i];
      const int r = u - pp.pre_rows[i];
      const size_t bb = it.L.block_bytes(), cs = (size_t)it.L.n_groups() * NVG;
      SpmmArgs a = it.sa;
      a.w = it.blk + (size_t)(j - 1) * bb;
      a.w_prev = j > 1 ? it.blk + (size_t)(j - 2) * bb : nullptr;
      a.z = it.blk + (size_t)j * bb;
      a.mz = it.coef + (size_t)j * cs;
      a.cp = it.coef + (size_t)(it.k + 2) * cs + (size_t)j * cs;
      const TermsSmem<T> terms = load_terms<T>(a.flips, a.n_flip, a.diags, a.n_diag);
      spmm_block<T, DS, VW, kModePass1, true>(it.L, a, terms, r % it.L.gridx, r / it.L.gridx, it.L.gridx);
      __syncthreads();  // the next unit rewrites the term tables
    }
    if (!grid_barrier(pp.bar, gen)) return;
    // phase B: A_j and Cw_j per bath vector
    for (int u = blockIdx.x; u < pp.pre_groups[na]; u += gridDim.x) {
      const int i = packed_item_of(pp.pre_groups, na, u);
      const PackedItem& it = pp.items[i];
      const size_t cs = (size_t)it.L.n_groups() * NVG;
      small_a_group<DS>(it.L, it.sa.partials, it.coef + (size_t)j * cs, it.ta + (size_t)(j - 1) * cs,
                        it.coef + (size_t)2 * (it.k + 2) * cs + (size_t)j * cs, it.flags, u - pp.pre_groups[i]);
      __syncthreads();
    }
    if (!grid_barrier(pp.bar, gen)) return;
    // phase C: W_{j+1} = Z + W_j Cw_j in place, partial sums of W_{j+1}^T W_{j+1}
    for (int u = blockIdx.x; u < pp.pre_rows[na]; u += gridDim.x) {
      const int i = packed_item_of(pp.pre_rows, na, u);
      const PackedItem& it = pp.items[i];
      const int r = u - pp.pre_rows[i];
      const size_t bb = it.L.block_bytes(), cs = (size_t)it.L.n_groups() * NVG;
      orth_block<T, DS, VW, true, true>(it.L, reinterpret_cast<const T*>(it.blk + (size_t)(j - 1) * bb),
                                        reinterpret_cast<T*>(it.blk + (size_t)j * bb),
                                        it.coef + (size_t)2 * (it.k + 2) * cs + (size_t)j * cs, it.sa.partials,
                                        nullptr, nullptr, 0, r % it.L.gridx, r / it.L.gridx, it.L.gridx);
      __syncthreads();
    }
    if (!grid_barrier(pp.bar, gen)) return;
    // phase D: Cholesky QR with deflation -> B_j, M_{j+1}, Cp_{j+1}
    for (int u = blockIdx.x; u < pp.pre_groups[na]; u += gridDim.x) {
      const int i = packed_item_of(pp.pre_groups, na, u);
      const PackedItem& it = pp.items[i];
      const size_t cs = (size_t)it.L.n_groups() * NVG;
      small_b_group<DS>(it.L, it.sa.partials, it.coef + (size_t)j * cs, it.tb + (size_t)(j - 1) * cs,
                        it.coef + (size_t)(j + 1) * cs, it.coef + (size_t)(it.k + 2) * cs + (size_t)(j + 1) * cs,
                        it.thr_abs_sq, it.thr_rel_sq, it.n_rec, it.flags, u - pp.pre_groups[i]);
      __syncthreads();
    }
    if (!grid_barrier(pp.bar, gen)) return;
  }
}

// The first pass of k_pass1_packed for one slice of one item per block: the recurrences
// of a slice's bath vectors read and write nothing of other slices, so the block runs
// every phase of every step for its slice alone -- the same row-block units and group
// units as the packed launch, in order, with block barriers between phases.
template <typename T, int DS, int VW>
__global__ void __launch_bounds__(kThreads) k_pass1_local(PackedPlan pp) {
  constexpr int NVG = DS * DS;
  const int u = blockIdx.x;
  const int i = packed_item_of(pp.pre_slices, pp.n_items, u);
  const PackedItem& it = pp.items[i];
  const int sl = u - pp.pre_slices[i];
  const size_t bb = it.L.block_bytes(), cs = (size_t)it.L.n_groups() * NVG;
  const int gx = it.L.gridx, gs = it.L.groups_per_slice();
  const TermsSmem<T> terms = load_terms<T>(it.sa.flips, it.sa.n_flip, it.sa.diags, it.sa.n_diag);
  for (int j = 1; j <= it.k; ++j) {
    SpmmArgs a = it.sa;
    a.w = it.blk + (size_t)(j - 1) * bb;
    a.w_prev = j > 1 ? it.blk + (size_t)(j - 2) * bb : nullptr;
    a.z = it.blk + (size_t)j * bb;
    a.mz = it.coef + (size_t)j * cs;
    a.cp = it.coef + (size_t)(it.k + 2) * cs + (size_t)j * cs;
    for (int bx = 0; bx < gx; ++bx) {
      spmm_block<T, DS, VW, kModePass1, true>(it.L, a, terms, bx, sl, gx);
      __syncthreads();
    }
    for (int g = 0; g < gs; ++g) {
      small_a_group<DS>(it.L, it.sa.partials, it.coef + (size_t)j * cs, it.ta + (size_t)(j - 1) * cs,
                        it.coef + (size_t)2 * (it.k + 2) * cs + (size_t)j * cs, it.flags, sl * gs + g);
      __syncthreads();
    }
    for (int bx = 0; bx < gx; ++bx) {
      orth_block<T, DS, VW, true, true>(it.L, reinterpret_cast<const T*>(it.blk + (size_t)(j - 1) * bb),
                                        reinterpret_cast<T*>(it.blk + (size_t)j * bb),
                                        it.coef + (size_t)2 * (it.k + 2) * cs + (size_t)j * cs, it.sa.partials,
                                        nullptr, nullptr, 0, bx, sl, gx);
      __syncthreads();
    }
    for (int g = 0; g < gs; ++g) {
      small_b_group<DS>(it.L, it.sa.partials, it.coef + (size_t)j * cs, it.tb + (size_t)(j - 1) * cs,
                        it.coef + (size_t)(j + 1) * cs, it.coef + (size_t)(it.k + 2) * cs + (size_t)(j + 1) * cs,
                        it.thr_abs_sq, it.thr_rel_sq, it.n_rec, it.flags, sl * gs + g);
      __syncthreads();
    }
  }
}

// ---------------------------------------------------------------- first pass in a cluster
//
// The whole first pass of one slice (float32, 2^kTileBits states per block) in one
// thread-block cluster: block `rank` keeps tile `rank` of W_j, and of W_{j-1}, in its shared
// memory for all k steps, reads partner tiles from the other blocks' shared memory, and the
// partial sums of A_j and of the QR Gram are exchanged the same way. A slice's recurrences
// read nothing of other slices, so no step needs more than two cluster barriers; every block
// of a cluster passes the same ones (k is the slice's), so each of them ends. Stored bases
// are written to global memory as they are formed. Every row's arithmetic is the tiled
// SpMM's and the orthogonalisation's, in their order (pass 2 recomputes the same bits).
//
// Bound by latency and the terms' shared-memory loads; two blocks per SM (at 128 registers,
// some spilled) hide more of it than one. It replaces, for batches, the untiled units of
// k_pass1_packed on items of 2^10 .. 2^14 states, which read every partner row from L2: the
// first passes of 48 small solves (N 8-14) take 44 instead of 87 ms.
constexpr int kClusterThreads = kConsumerWarps * 32;

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}
// The same shared-memory address in block `rank` of the cluster.
template <typename P>
__device__ __forceinline__ const P* peer(const P* p, uint32_t rank) {
  uint64_t r;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
  return reinterpret_cast<const P*>(r);
}

__host__ __device__ inline size_t cluster_smem_bytes(const TiledTerms& tt) {
  return 2 * (size_t)kTileBytes + 8 * 32 * sizeof(double) + (size_t)kConsumerWarps * 2 * 16 * sizeof(double) +
         (size_t)tt.n_part * sizeof(PatS<float>) + (size_t)tt.n_grp * sizeof(GrpS<float>) +
         (size_t)tt.n_lane * sizeof(LaneS<float>) +
         sizeof(float) * (16 + 4 * 32 + kTileRows + (size_t)tile_diag_stride(tt.dg.n_entries, 4)) + 64;
}

template <int DS>
__global__ void __launch_bounds__(kClusterThreads, 2) k_pass1_cluster(PackedPlan pp, int c_log) {
  using T = float;
  constexpr int VW = 4, LPR = 2, BS = VW * LPR, RG = kClusterThreads / LPR, RPT = kTileRows / RG;
  constexpr int kStep = RG * BS, kTile = kTileRows * BS;
  constexpr int NG = VW / DS, NVG = DS * DS, NV = NG * NVG;
  constexpr int GS = LPR * NG, GV = GS * NVG;  // groups of the slice and their values
  const uint32_t rank = blockIdx.x & ((1u << c_log) - 1u), peers = 1u << c_log;
  const int u = blockIdx.x >> c_log;
  const int item = packed_item_of(pp.pre_slices, pp.n_items, u);
  const PackedItem& it = pp.items[item];
  const int slice = u - pp.pre_slices[item];
  const TiledTerms& tt = it.sa.tiled;
  extern __shared__ __align__(128) unsigned char smem_c[];
  T* const buf = reinterpret_cast<T*>(smem_c);
  double* const sM = reinterpret_cast<double*>(buf + 2 * kTile);  // M_j of the slice's groups
  double* const sMn = sM + 32;
  double* const sCp = sM + 64;
  double* const sTot = sM + 96;
  double* const sA = sM + 128;
  double* const sR = sM + 160;
  double* const part_a = sM + 192;  // this block's sums of W_j^T Z ...
  double* const part_b = sM + 224;  // ... and of W_{j+1}^T W_{j+1}
  double* const red = sM + 256;     // [warp][lane][NV]
  PatS<T>* const pat = reinterpret_cast<PatS<T>*>(red + kConsumerWarps * 2 * 16);
  GrpS<T>* const grp = reinterpret_cast<GrpS<T>*>(pat + tt.n_part);
  LaneS<T>* const lanet = reinterpret_cast<LaneS<T>*>(grp + tt.n_grp);
  T* const s_reg = reinterpret_cast<T*>(lanet + tt.n_lane);
  T* const s_mz = s_reg + 16;
  T* const s_cp = s_mz + 32;
  T* const s_cw = s_cp + 32;
  T* const s_low = s_cw + 64;
  T* const s_hk = s_low + kTileRows;

  load_tables<BS>(tt, pat, grp, lanet, s_reg, s_low);
  const int hstride = tile_diag_stride(tt.dg.n_entries, (int)sizeof(T));
  for (int i = threadIdx.x; i < hstride; i += kClusterThreads)
    s_hk[i] = reinterpret_cast<const T*>(it.sa.tile_k)[(size_t)rank * hstride + i];
  const int lane = threadIdx.x % LPR, rg = threadIdx.x / LPR, warp = threadIdx.x >> 5;
  const int rgoff = rg * BS + lane * VW;
  const size_t bb = it.L.block_bytes(), cs = (size_t)it.L.n_groups() * NVG, go = (size_t)slice * GV;
  // this thread's first row in block 0 of the basis
  const size_t row_b = ((size_t)slice * it.L.D * BS + (size_t)rank * kTile + rgoff) * sizeof(T);
  T xo[RPT][VW];
  load_rows<kStep>(xo, reinterpret_cast<const T*>(it.blk + row_b));
#pragma unroll
  for (int m = 0; m < RPT; ++m) VecIO<T, VW>::st(buf + rgoff + m * kStep, xo[m]);
  if (threadIdx.x < GV) {
    sM[threadIdx.x] = it.coef[cs + go + threadIdx.x];
    s_mz[threadIdx.x] = (T)sM[threadIdx.x];
    s_cp[threadIdx.x] = (T)0;
  }
  __syncthreads();
  uint32_t act_lane = 0u, act_grp = 0u;
  for (int t = 0; t < tt.n_own; ++t) act_lane |= (uint32_t)(__popc((uint32_t)rg & lanet[t].low) & 1) << t;
  for (int t = 0; t < tt.n_grp; ++t) act_grp |= (uint32_t)(((uint32_t)rg & grp[t].low) != 0u) << t;
  // patterns whose high spin is up (bit p) in this block's tile
  uint32_t up_pairs = 0u;
  for (int p = 0; p < tt.n_pair; ++p) up_pairs |= (uint32_t)((rank & pat[p].high) != 0u) << p;
  cluster_sync();

  // The block's sums of NV values per thread over the threads of a lane: out[lane][NV].
  auto block_sums = [&](const T* vals, double* out) {
#pragma unroll
    for (int e = 0; e < NV; ++e) {
      T x = vals[e];
#pragma unroll
      for (int o = LPR; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
      if ((threadIdx.x & 31) < LPR) red[(warp * LPR + lane) * 16 + e] = (double)x;
    }
    __syncthreads();
    if (threadIdx.x < GV) {
      const int ln = threadIdx.x / NV, e = threadIdx.x % NV;
      double sum = 0.0;
      for (int w = 0; w < kConsumerWarps; ++w) sum += red[(w * LPR + ln) * 16 + e];
      out[threadIdx.x] = sum;
    }
  };
  // The cluster's sums of part (after a cluster barrier), the blocks in order.
  auto cluster_sums = [&](const double* part) {
    if (threadIdx.x < GV) {
      double sum = 0.0;
      for (uint32_t r = 0; r < peers; ++r) sum += peer(part, r)[threadIdx.x];
      sTot[threadIdx.x] = sum;
    }
    __syncthreads();
  };

  for (int j = 1; j <= it.k; ++j) {
    const T* const cur = buf + ((j - 1) & 1) * kTile;  // W_j
    T* const oth = buf + (j & 1) * kTile;              // W_{j-1}, then W_{j+1}
    T y[RPT][VW];
    {
      T dg[RPT];
      tile_diagonal<T, RPT, RG>(dg, s_low, s_hk, rg, tt.dg);
#pragma unroll
      for (int m = 0; m < RPT; ++m)
#pragma unroll
        for (int v = 0; v < VW; ++v) y[m][v] = dg[m] * xo[m][v];
    }
    own_terms<false, false, RG, kStep>(y, xo, cur, rgoff, tt, s_reg, grp, lanet, act_lane, act_grp);
    // partner tiles in the tiled SpMM's order
    uint32_t om = up_pairs, zm = ~up_pairs & (uint32_t)((1u << tt.n_pair) - 1u);
    for (int joint = min(__popc(zm), __popc(om)); zm | om; --joint) {
      if (joint > 0) {
        const int z = __ffs((int)zm) - 1, o = __ffs((int)om) - 1;
        zm &= zm - 1u;
        om &= om - 1u;
        pair_terms<kStep>(y, peer(cur, rank ^ pat[z].high), peer(cur, rank ^ pat[o].high), rgoff, rg, pat[z], pat[o],
                          lanet);
      } else {
        const int p = __ffs((int)(zm | om)) - 1;
        zm &= ~(1u << p);
        om &= ~(1u << p);
        single_terms<false, false, kStep>(y, peer(cur, rank ^ pat[p].high), rgoff, rg, pat[p], (rank & pat[p].high) != 0u, lanet);
      }
    }
    for (int p = tt.n_pair; p < tt.n_pair + tt.n_single; ++p)
      single_terms<false, false, kStep>(y, peer(cur, rank ^ pat[p].high), rgoff, rg, pat[p], (rank & pat[p].high) != 0u, lanet);
    for (int p = tt.n_pair + tt.n_single; p < tt.n_part; ++p) {
      const T c = (__popc(rank & pat[p].high) & 1) ? pat[p].co[0] : pat[p].ce[0];
      if (in_use(c)) rows_fma<kStep>(y, peer(cur, rank ^ pat[p].high) + rgoff, c);
    }
    // Z = (H W_j) M_j + W_{j-1} Cp_j into y, and the sums of W_j^T Z
    T vals[NV];
#pragma unroll
    for (int e = 0; e < NV; ++e) vals[e] = (T)0;
    {
      T mz[NV], cp[NV];
#pragma unroll
      for (int e = 0; e < NV; ++e) {
        mz[e] = s_mz[lane * NV + e];
        cp[e] = s_cp[lane * NV + e];
      }
#pragma unroll
      for (int m = 0; m < RPT; ++m) {
        T z[VW];
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int c = 0; c < DS; ++c) {
            T t = (T)0;
#pragma unroll
            for (int i = 0; i <= c; ++i) t = fma(y[m][g * DS + i], mz[g * NVG + i * DS + c], t);
            z[g * DS + c] = t;
          }
        if (j > 1) {
          T xp[VW];
          VecIO<T, VW>::ld_rw(xp, oth + rgoff + m * kStep);
#pragma unroll
          for (int g = 0; g < NG; ++g)
#pragma unroll
            for (int c = 0; c < DS; ++c) {
              T t = z[g * DS + c];
#pragma unroll
              for (int i = 0; i < DS; ++i) t = fma(xp[g * DS + i], cp[g * NVG + i * DS + c], t);
              z[g * DS + c] = t;
            }
        }
#pragma unroll
        for (int g = 0; g < NG; ++g)
#pragma unroll
          for (int i = 0; i < DS; ++i)
#pragma unroll
            for (int c = 0; c < DS; ++c)
              vals[g * NVG + i * DS + c] = fma(xo[m][g * DS + i], z[g * DS + c], vals[g * NVG + i * DS + c]);
#pragma unroll
        for (int v = 0; v < VW; ++v) y[m][v] = z[v];
      }
    }
    block_sums(vals, part_a);
    cluster_sync();
    cluster_sums(part_a);
    // A_j and Cw_j (small_a_group): thread e of the slice's values
    const int e = threadIdx.x, g = e / NVG, r = e % NVG / DS, c = e % DS;
    if (e < GV) {
      double p1 = 0.0, p2 = 0.0;  // (Q_j^T Z)[r][c] and [c][r]
      for (int i = 0; i < DS; ++i) {
        p1 += sM[g * NVG + i * DS + r] * sTot[g * NVG + i * DS + c];
        p2 += sM[g * NVG + i * DS + c] * sTot[g * NVG + i * DS + r];
      }
      sA[e] = 0.5 * (p1 + p2);
    }
    __syncthreads();
    if (e < GV) {
      double cw = 0.0;
      for (int i = 0; i < DS; ++i) cw += sM[g * NVG + r * DS + i] * sA[g * NVG + i * DS + c];
      s_cw[e] = (T)-cw;
      if (rank == 0) {
        it.ta[(size_t)(j - 1) * cs + go + e] = sA[e];
        it.coef[(size_t)2 * (it.k + 2) * cs + (size_t)j * cs + go + e] = -cw;
        if (!isfinite(sA[e])) atomicOr(it.flags, kFlagNonFinite);
      }
    }
    __syncthreads();
    // W_{j+1} = Z + W_j Cw_j, its sums, its rows kept
    {
      T cw[NV];
#pragma unroll
      for (int q = 0; q < NV; ++q) {
        cw[q] = s_cw[lane * NV + q];
        vals[q] = (T)0;
      }
      T* const out = reinterpret_cast<T*>(it.blk + (size_t)j * bb + row_b);
#pragma unroll
      for (int m = 0; m < RPT; ++m) {
#pragma unroll
        for (int q = 0; q < NG; ++q)
#pragma unroll
          for (int cc = 0; cc < DS; ++cc) {
            T t = y[m][q * DS + cc];
#pragma unroll
            for (int i = 0; i < DS; ++i) t = fma(xo[m][q * DS + i], cw[q * NVG + i * DS + cc], t);
            y[m][q * DS + cc] = t;
          }
#pragma unroll
        for (int q = 0; q < NG; ++q)
#pragma unroll
          for (int i = 0; i < DS; ++i)
#pragma unroll
            for (int cc = i; cc < DS; ++cc)
              vals[q * NVG + i * DS + cc] = fma(y[m][q * DS + i], y[m][q * DS + cc], vals[q * NVG + i * DS + cc]);
        VecIO<T, VW>::st(oth + rgoff + m * kStep, y[m]);
        VecIO<T, VW>::st_cs(out + m * kStep, y[m]);
#pragma unroll
        for (int v = 0; v < VW; ++v) xo[m][v] = y[m][v];
      }
#pragma unroll
      for (int q = 0; q < NG; ++q)
#pragma unroll
        for (int i = 0; i < DS; ++i)
#pragma unroll
          for (int cc = 0; cc < i; ++cc) vals[q * NVG + i * DS + cc] = vals[q * NVG + cc * DS + i];
    }
    block_sums(vals, part_b);
    cluster_sync();  // W_{j+1} and part_b of every block are there
    cluster_sums(part_b);
    // B_j, M_{j+1}, Cp_{j+1} (small_b_group): one thread per group
    if (threadIdx.x < GS) {
      const int o = threadIdx.x * NVG;
      bool finite;
      const bool dropped =
          qr_group<DS>(sTot + o, sM + o, it.thr_abs_sq, it.thr_rel_sq, sR + o, sMn + o, sCp + o, finite);
      if (rank == 0) {
        if (dropped && slice * GS + (int)threadIdx.x < it.n_rec) atomicOr(it.flags, (uint32_t)RDM_FLAG_DEFLATED);
        if (!finite) atomicOr(it.flags, kFlagNonFinite);
      }
    }
    __syncthreads();
    if (e < GV) {
      sM[e] = sMn[e];
      s_mz[e] = (T)sMn[e];
      s_cp[e] = (T)sCp[e];
      if (rank == 0) {
        it.tb[(size_t)(j - 1) * cs + go + e] = sR[e];
        it.coef[(size_t)(j + 1) * cs + go + e] = sMn[e];
        it.coef[(size_t)(it.k + 2) * cs + (size_t)(j + 1) * cs + go + e] = sCp[e];
      }
    }
    __syncthreads();
  }
  cluster_sync();  // no block leaves while another may still read its shared memory
}

inline dim3 grid_of(const Layout& L) { return dim3((unsigned)L.gridx, (unsigned)L.n_slices); }

template <typename T>
size_t terms_smem(int nf, int nd) {
  return (size_t)(2 * nf + nd) * sizeof(T) + (size_t)(nf + nd) * sizeof(uint32_t) + 16;
}

}  // namespace

// Raises a kernel's dynamic shared-memory limit to the device maximum (minus its
// static shared memory), once per kernel. Setting it to the largest value once,
// instead of to each launch's size, keeps concurrent host threads from lowering it
// under one another's launches.
static cudaError_t opt_in_smem(const void* func) {
  static std::mutex mu;
  static std::set<const void*> done;
  std::lock_guard<std::mutex> lk(mu);
  if (done.count(func)) return cudaSuccess;
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa{};
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, func);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             optin - (int)fa.sharedSizeBytes);
  if (e == cudaSuccess) done.insert(func);
  return e;
}

// ---------------------------------------------------------------- dispatch

#define RDM_DISPATCH(L, ...)                                         \
  do {                                                                \
    if ((L).precision == RDM_FP32) {                                  \
      using T = float;                                                \
      constexpr int VW = 4;                                           \
      if ((L).DS == 1) { constexpr int DS = 1; __VA_ARGS__; }                \
      else if ((L).DS == 2) { constexpr int DS = 2; __VA_ARGS__; }           \
      else { constexpr int DS = 4; __VA_ARGS__; }                            \
    } else {                                                          \
      using T = double;                                               \
      if ((L).DS == 1) { constexpr int DS = 1; constexpr int VW = 2; __VA_ARGS__; } \
      else if ((L).DS == 2) { constexpr int DS = 2; constexpr int VW = 2; __VA_ARGS__; } \
      else { constexpr int DS = 4; constexpr int VW = 4; __VA_ARGS__; }      \
    }                                                                 \
  } while (0)

#define RDM_DISPATCH_DS(DSV, ...)                      \
  do {                                                  \
    if ((DSV) == 1) { constexpr int DS = 1; __VA_ARGS__; }     \
    else if ((DSV) == 2) { constexpr int DS = 2; __VA_ARGS__; } \
    else { constexpr int DS = 4; __VA_ARGS__; }                \
  } while (0)

cudaError_t launch_gauss_norms(int64_t d_b, int n_v, uint64_t seed, int64_t l0, double* partials,
                               double* inv_norm, cudaStream_t st, double* graw) {
  int gx = (int)((d_b + 4095) / 4096);
  if (gx > 64) gx = 64;
  if (gx < 1) gx = 1;
  k_gauss_sumsq<<<dim3(gx, n_v), kThreads, 0, st>>>(d_b, seed, l0, partials, graw);
  k_gauss_finish<<<(n_v + 127) / 128, 128, 0, st>>>(n_v, gx, partials, inv_norm);
  return cudaGetLastError();
}

cudaError_t launch_init_block(const Layout& L, int dist, uint64_t seed, int64_t l0, int n_v_real,
                              const double* inv_norm, const void* vbuf, void* W, cudaStream_t st,
                              int sub, const BathPerm* bp) {
  BathPerm id{};
  const BathPerm perm = bp ? *bp : id;
  if (perm.n < 0 || perm.n > L.n_bath_bits) return cudaErrorInvalidValue;
  for (int q = 0; q < perm.n; ++q)
    if (perm.src[q] >= perm.n) return cudaErrorInvalidValue;
  RDM_DISPATCH(L, (k_init_block<T, DS, VW><<<grid_of(L), kThreads, 0, st>>>(
                      L, dist, seed, l0, n_v_real, inv_norm, reinterpret_cast<const T*>(vbuf),
                      reinterpret_cast<T*>(W), sub, perm)));
  return cudaGetLastError();
}

cudaError_t launch_gauss_fill(const Layout& L, int n_v, uint64_t seed, int64_t l0,
                              const double* inv_norm, void* vbuf, cudaStream_t st, const double* graw) {
  const int64_t d_b = int64_t(1) << L.n_bath_bits;
  int gx = (int)std::min<int64_t>((d_b + 255) / 256, 1024);
  k_gauss_fill<<<dim3(gx, n_v), 256, 0, st>>>(d_b, seed, l0, inv_norm, graw, L.precision, vbuf);
  return cudaGetLastError();
}

cudaError_t launch_tile_diag(const Layout& L, const TileDiag& dg, void* out, cudaStream_t st) {
  const int64_t tiles = L.D >> kTileBits;
  const int stride = tile_diag_stride(dg.n_entries, L.elem);
  const int gx = (int)std::min<int64_t>(tiles, 4096);
  const size_t sm = (size_t)(dg.n_groups + 1) * sizeof(double);
  if (sm > 48 * 1024) return cudaErrorInvalidValue;
  if (L.precision == RDM_FP32)
    k_tile_diag<float><<<gx, kThreads, sm, st>>>(tiles, dg, stride, reinterpret_cast<float*>(out));
  else
    k_tile_diag<double><<<gx, kThreads, sm, st>>>(tiles, dg, stride, reinterpret_cast<double*>(out));
  return cudaGetLastError();
}

// Runs of 2^r consecutive tiles per block: a block closes its partial sums and loads the
// mixing coefficients at every change of slice, which costs about a third of a tile's time,
// so slices of few tiles (N = 16: 64 tiles, fewer than the 152 blocks) are walked in runs.
// The r with the smallest largest block, counting that; 0 for slices of many tiles.
static int tiled_run_log(const Layout& L) {
  const int64_t per = L.D >> kTileBits, total = per * L.n_slices, grid = spmm_tiled_grid(L);
  int best = 0;
  double least = 1e300;
  for (int r = 0; r <= 3 && (1 << r) <= per; ++r) {
    const int64_t runs = total >> r, mine = (runs + grid - 1) / grid;
    // slices a block enters: one per run, or per pass over a slice longer than the stride
    const double slices = std::min<double>((double)mine, (double)(mine * grid << r) / (double)per + 1.0);
    const double cost = (double)(mine << r) + 0.35 * slices;
    if (cost < 0.999 * least) {
      least = cost;
      best = r;
    }
  }
  return best;
}

template <typename T, int DS, int MODE, bool UNI, bool TILE_SUMS>
static cudaError_t launch_tiled_sums(const Layout& L, const SpmmArgs& a0, int run_log, cudaStream_t st) {
  cudaError_t e = opt_in_smem(reinterpret_cast<const void*>(k_spmm_tiled<T, DS, MODE, UNI, TILE_SUMS>));
  if (e != cudaSuccess) return e;
  static int optin = 0;
  if (!optin) {
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e != cudaSuccess) return e;
  }
  // Deepest ring (up to 6 slots) that fits beside this Hamiltonian's term tables.
  SpmmArgs a = a0;
  a.run_log = run_log;
  const TiledTerms& tt = a.tiled;
  a.stages = 6;  // a multiple of kProducerWarps
  while (a.stages > kProducerWarps &&
         tiled_smem_bytes<T>(tt.n_part, tt.n_lane, tt.n_grp, tt.dg.n_entries, a.stages) > (size_t)optin)
    a.stages -= kProducerWarps;
  const size_t sm = tiled_smem_bytes<T>(tt.n_part, tt.n_lane, tt.n_grp, tt.dg.n_entries, a.stages);
  if (sm > (size_t)optin) return cudaErrorInvalidValue;
  k_spmm_tiled<T, DS, MODE, UNI, TILE_SUMS><<<dim3((unsigned)spmm_tiled_grid(L), 1), kTiledThreads, sm, st>>>(L, a);
  return cudaGetLastError();
}

template <typename T, int DS, int MODE, bool UNI = false>
static cudaError_t launch_tiled(const Layout& L, const SpmmArgs& a, cudaStream_t st) {
  const int run_log = tiled_run_log(L);
  constexpr bool kSums = MODE == kModePass1 && sizeof(T) == 4;
  if constexpr (kSums && UNI)
    if (run_log == 0) return launch_tiled_sums<T, DS, MODE, UNI, false>(L, a, run_log, st);
  return launch_tiled_sums<T, DS, MODE, UNI, kSums>(L, a, run_log, st);
}

cudaError_t launch_spmm(const Layout& L, int mode, const SpmmArgs& a, cudaStream_t st) {
  if (layout_tiled(L) && a.tiled.ready && a.tile_k) {
    const bool f32 = L.precision == RDM_FP32;
    if (mode == kModeApply) {
      if (L.DS != 1) return cudaErrorInvalidValue;
      return f32 ? launch_tiled<float, 1, kModeApply>(L, a, st) : launch_tiled<double, 1, kModeApply>(L, a, st);
    }
    // UNI: no parity-dependent coefficient anywhere
    const bool uni = a.tiled.all_uniform != 0, p1 = mode == kModePass1;
    auto go = [&](auto t, auto ds) -> cudaError_t {
      using T = decltype(t);
      constexpr int DS = decltype(ds)::value;
      if (uni) return p1 ? launch_tiled<T, DS, kModePass1, true>(L, a, st) : launch_tiled<T, DS, kModePass2, true>(L, a, st);
      return p1 ? launch_tiled<T, DS, kModePass1>(L, a, st) : launch_tiled<T, DS, kModePass2>(L, a, st);
    };
    auto by_ds = [&](auto t) -> cudaError_t {
      if (L.DS == 1) return go(t, std::integral_constant<int, 1>{});
      if (L.DS == 2) return go(t, std::integral_constant<int, 2>{});
      return go(t, std::integral_constant<int, 4>{});
    };
    return f32 ? by_ds(float{}) : by_ds(double{});
  }
  RDM_DISPATCH(L, {
    const size_t sm = terms_smem<T>(a.n_flip, a.n_diag);
    if (mode == kModeApply)
      k_spmm<T, DS, VW, kModeApply><<<grid_of(L), kThreads, sm, st>>>(L, a);
    else if (mode == kModePass1)
      k_spmm<T, DS, VW, kModePass1><<<grid_of(L), kThreads, sm, st>>>(L, a);
    else
      k_spmm<T, DS, VW, kModePass2><<<grid_of(L), kThreads, sm, st>>>(L, a);
  });
  return cudaGetLastError();
}

cudaError_t launch_orth(const Layout& L, const void* w, void* z, const double* cw,
                        double* partials, cudaStream_t st) {
  RDM_DISPATCH(L, (k_orth<T, DS, VW, true><<<grid_of(L), kThreads, 0, st>>>(
                      L, reinterpret_cast<const T*>(w), reinterpret_cast<T*>(z), cw, partials,
                      nullptr, nullptr, 0)));
  return cudaGetLastError();
}

cudaError_t launch_orth_psi(const Layout& L, const void* w, void* z, const double* cw, void* psi,
                            const double* e, int nb, cudaStream_t st) {
  RDM_DISPATCH(L, {
    const size_t sm = (size_t)nb * L.groups_per_slice() * DS * DS * sizeof(T) + 16;
    cudaError_t ce = opt_in_smem(reinterpret_cast<const void*>(k_orth<T, DS, VW, false>));
    if (ce != cudaSuccess) return ce;
    k_orth<T, DS, VW, false><<<grid_of(L), kThreads, sm, st>>>(
        L, reinterpret_cast<const T*>(w), reinterpret_cast<T*>(z), cw, nullptr,
        reinterpret_cast<T*>(psi), e, nb);
  });
  return cudaGetLastError();
}

cudaError_t launch_psi_batch(const Layout& L, const PsiBatch& wb, int m, void* psi, const double* e,
                             size_t estride, int nb, cudaStream_t st) {
  if (m < 1 || m > kPsiBatchMax) return cudaErrorInvalidValue;
  RDM_DISPATCH(L, {
    const size_t sm = (size_t)m * nb * L.groups_per_slice() * DS * DS * sizeof(T) + 16;
    cudaError_t ce = opt_in_smem(reinterpret_cast<const void*>(k_psi_batch<T, DS, VW>));
    if (ce != cudaSuccess) return ce;
    k_psi_batch<T, DS, VW><<<grid_of(L), kThreads, sm, st>>>(L, wb, m, reinterpret_cast<T*>(psi), e, estride,
                                                             nb);
  });
  return cudaGetLastError();
}

cudaError_t launch_psi_init(const Layout& L, const void* w, void* psi, const double* e, int nb,
                            cudaStream_t st) {
  RDM_DISPATCH(L, (k_psi_init<T, DS, VW><<<grid_of(L), kThreads, 0, st>>>(
                      L, reinterpret_cast<const T*>(w), reinterpret_cast<T*>(psi), e, nb)));
  return cudaGetLastError();
}

cudaError_t launch_coef_init(const Layout& L, StepCoefs c1, cudaStream_t st) {
  const int ng = L.n_groups();
  RDM_DISPATCH_DS(L.DS, (k_coef_init<DS><<<(ng + 127) / 128, 128, 0, st>>>(ng, c1.mz, c1.cp)));
  return cudaGetLastError();
}

cudaError_t launch_small_a(const Layout& L, const double* partials, const double* mz,
                           double* a_out, double* cw_out, uint32_t* flags, cudaStream_t st) {
  RDM_DISPATCH_DS(L.DS, (k_small_a<DS><<<L.n_groups(), kSmallThreads, 0, st>>>(
                           L, partials, mz, a_out, cw_out, flags)));
  return cudaGetLastError();
}

cudaError_t launch_small_b(const Layout& L, const double* partials, const double* mz_j,
                           double* b_out, double* mz_next, double* cp_next, double thr_abs_sq,
                           double thr_rel_sq, int n_groups_real, uint32_t* flags,
                           cudaStream_t st) {
  RDM_DISPATCH_DS(L.DS, (k_small_b<DS><<<L.n_groups(), kSmallThreads, 0, st>>>(
                           L, partials, mz_j, b_out, mz_next, cp_next, thr_abs_sq, thr_rel_sq,
                           n_groups_real, flags)));
  return cudaGetLastError();
}

template <typename T, int DS, int VW>
static cudaError_t packed_kernel_info(const void** fn) {
  *fn = reinterpret_cast<const void*>(k_pass1_packed<T, DS, VW>);
  return opt_in_smem(*fn);
}

static cudaError_t packed_fn(int precision, int ds, const void** fn) {
  Layout L{};
  L.precision = precision;
  L.DS = ds;
  cudaError_t e = cudaErrorInvalidValue;
  RDM_DISPATCH(L, e = (packed_kernel_info<T, DS, VW>(fn)));
  return e;
}

size_t spmm_terms_smem(int precision, int n_flip, int n_diag) {
  return precision == RDM_FP32 ? terms_smem<float>(n_flip, n_diag) : terms_smem<double>(n_flip, n_diag);
}

int packed_max_blocks_per_sm(int precision, int ds, size_t smem) {
  const void* fn = nullptr;
  if (packed_fn(precision, ds, &fn) != cudaSuccess) return 0;
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, kThreads, smem) != cudaSuccess) return 0;
  return n;
}

template <typename T, int DS, int VW>
static cudaError_t local_kernel_info(const void** fn) {
  *fn = reinterpret_cast<const void*>(k_pass1_local<T, DS, VW>);
  return opt_in_smem(*fn);
}

cudaError_t launch_pass1_local(int precision, int ds, const PackedPlan& pp, int grid, size_t smem,
                               cudaStream_t st) {
  Layout L{};
  L.precision = precision;
  L.DS = ds;
  const void* fn = nullptr;
  cudaError_t e = cudaErrorInvalidValue;
  RDM_DISPATCH(L, e = (local_kernel_info<T, DS, VW>(&fn)));
  if (e != cudaSuccess) return e;
  PackedPlan arg = pp;
  void* args[] = {&arg};
  return cudaLaunchKernel(fn, dim3((unsigned)grid), dim3(kThreads), args, smem, st);
}

// One launch of k_pass1_cluster<DS>: `at` is its attribute storage.
template <int DS>
static cudaError_t cluster_launch(int c_log, int n_slices, size_t smem, cudaStream_t st, cudaLaunchAttribute* at,
                                  cudaLaunchConfig_t* cfg) {
  const void* fn = reinterpret_cast<const void*>(k_pass1_cluster<DS>);
  cudaError_t e = opt_in_smem(fn);
  // (16 blocks exceed the portable cluster size)
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)n_slices << c_log);
  cfg->blockDim = dim3(kClusterThreads);
  cfg->dynamicSmemBytes = smem;
  cfg->stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = 1u << c_log;
  at->val.clusterDim.y = at->val.clusterDim.z = 1;
  cfg->attrs = at;
  cfg->numAttrs = 1;
  return e;
}

// More than any item of up to 2^14 states needs (about 80 KB).
constexpr size_t kClusterSmemMax = (size_t)96 * 1024;

// Whether the device can hold a cluster of 2^c_log blocks of k_pass1_cluster<ds> (a device
// partition of few SMs, or no device, cannot); asked once per device, d_s and size.
static bool device_takes_cluster(int ds, int c_log) {
  static std::mutex mu;
  static std::map<std::array<int, 3>, bool> known;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  std::lock_guard<std::mutex> lk(mu);
  const std::array<int, 3> key{dev, ds, c_log};
  const auto f = known.find(key);
  if (f != known.end()) return f->second;
  auto ask = [&](auto d) -> bool {
    constexpr int DS = decltype(d)::value;
    cudaLaunchAttribute at{};
    cudaLaunchConfig_t cfg;
    int n = 0;
    cudaError_t e = cluster_launch<DS>(c_log, 1, kClusterSmemMax, nullptr, &at, &cfg);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, k_pass1_cluster<DS>, &cfg);
    if (e != cudaSuccess) cudaGetLastError();
    return e == cudaSuccess && n > 0;
  };
  const bool ok = ds == 1   ? ask(std::integral_constant<int, 1>{})
                  : ds == 2 ? ask(std::integral_constant<int, 2>{})
                            : ask(std::integral_constant<int, 4>{});
  known[key] = ok;
  return ok;
}

bool pass1_cluster_fits(const Layout& L, const TiledTerms& tt) {
  const int c_log = L.n_bits - kTileBits;
  return L.precision == RDM_FP32 && layout_tiled(L) && tt.ready && c_log <= kClusterMaxLog &&
         cluster_smem_bytes(tt) <= kClusterSmemMax && device_takes_cluster(L.DS, c_log);
}

cudaError_t launch_pass1_cluster(int ds, const PackedPlan& pp, int c_log, int n_slices, size_t smem, cudaStream_t st) {
  if (c_log < 0 || c_log > kClusterMaxLog) return cudaErrorInvalidValue;
  auto go = [&](auto d) -> cudaError_t {
    constexpr int DS = decltype(d)::value;
    cudaLaunchAttribute at{};
    cudaLaunchConfig_t cfg;
    const cudaError_t e = cluster_launch<DS>(c_log, n_slices, smem, st, &at, &cfg);
    return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, k_pass1_cluster<DS>, pp, c_log) : e;
  };
  if (ds == 1) return go(std::integral_constant<int, 1>{});
  if (ds == 2) return go(std::integral_constant<int, 2>{});
  return go(std::integral_constant<int, 4>{});
}

size_t pass1_cluster_smem(const TiledTerms& tt) { return cluster_smem_bytes(tt); }

cudaError_t launch_pass1_packed(int precision, int ds, const PackedPlan& pp, int grid, size_t smem,
                                cudaStream_t st) {
  const void* fn = nullptr;
  cudaError_t e = packed_fn(precision, ds, &fn);
  if (e != cudaSuccess) return e;
  PackedPlan arg = pp;
  void* args[] = {&arg};
  return cudaLaunchCooperativeKernel(fn, dim3((unsigned)grid), dim3(kThreads), args, smem, st);
}

static bool gram_on_rows(const Layout& L) { return L.precision == RDM_FP32 && layout_tiled(L); }

int gram_gridx(const Layout& L) {
  if (!gram_on_rows(L)) return L.gridx;
  // about 3 blocks per SM (what is resident) and beta group over all slices
  const int64_t chunks = L.D / kGramChunk;
  return (int)std::max<int64_t>(1, std::min<int64_t>(chunks, 456 / L.n_slices));
}

template <int DS, int NBT, bool FINAL>
static cudaError_t launch_gram_rows(const Layout& L, const float* w, const GramBetas& gb, int k, const double* e,
                                    int nbs, int b0, int nb, int nz, double* partials, size_t pstride, cudaStream_t st) {
  cudaError_t ce = opt_in_smem(reinterpret_cast<const void*>(k_gram_rows<DS, NBT, FINAL>));
  if (ce != cudaSuccess) return ce;
  const size_t sm = (size_t)kGramStages * (NBT >= 4 ? 2 : 4) * kGramThreads * 16 +
                    (FINAL ? 0 : (size_t)k * NBT * 8 * DS * sizeof(float));
  k_gram_rows<DS, NBT, FINAL><<<dim3((unsigned)(L.gridx * nz), (unsigned)L.n_slices), kGramThreads, sm, st>>>(
      L, w, gb, e, nbs, b0, nb, nz, partials, pstride);
  return cudaGetLastError();
}

cudaError_t launch_final_gram(const Layout& L, const void* psi, int nb, double* partials, size_t pstride,
                              cudaStream_t st) {
  if (gram_on_rows(L)) {
    const GramBetas gb{};
    const float* w = reinterpret_cast<const float*>(psi);
    RDM_DISPATCH_DS(L.DS, return (launch_gram_rows<DS, 1, true>(L, w, gb, 0, nullptr, 0, 0, nb, nb, partials,
                                                                pstride, st)));
  }
  for (int b = 0; b < nb; ++b)
    RDM_DISPATCH(L, (k_final_gram<T, DS, VW><<<grid_of(L), kThreads, 0, st>>>(
                        L, reinterpret_cast<const T*>(psi) + (size_t)b * L.D * L.B, partials + b * pstride)));
  return cudaGetLastError();
}

// The betas b0 .. b0+nb-1 in nz groups (kb: the last step of each) of at most 4 (8 leave
// 2 blocks per SM for d_s = 2 and run 5% slower) whose coefficients of k steps take at most
// 36 KB: with a group of 4, whose ring is 32 KB, 3 blocks per SM. Groups of 2 and 1 hold 4 rows
// a thread and a ring of 64 KB: 3 blocks per SM up to 10 KB of coefficients, 2 beyond (d_s = 4
// grids of k > 72; N = 14, n_v = 64, 8 betas, k = 100: 14.2 ms a solve, 27.8 with k_gram_stored).
template <int DS>
static cudaError_t launch_gram_groups(const Layout& L, const float* w, int k, const int* kb, const double* e, int nbs,
                                      int b0, int nb, double* partials, size_t pstride, cudaStream_t st) {
  if (nb > kGramLaunchBetas) return cudaErrorInvalidValue;
  int most = 4;
  while (most > 1 && (size_t)k * most * 8 * DS * sizeof(float) > ((size_t)36 << 10)) most /= 2;
  const int nz = (nb + most - 1) / most, group = (nb + nz - 1) / nz;
  std::vector<int> ord(nb);
  for (int b = 0; b < nb; ++b) ord[b] = b;
  std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return kb[x] > kb[y]; });
  GramBetas gb{};
  for (int q = 0; q < nb; ++q) {
    gb.k[q] = (uint16_t)kb[ord[q]];
    gb.beta[q] = (uint8_t)ord[q];
  }
  if (group > 2) return launch_gram_rows<DS, 4, false>(L, w, gb, k, e, nbs, b0, nb, nz, partials, pstride, st);
  if (group > 1) return launch_gram_rows<DS, 2, false>(L, w, gb, k, e, nbs, b0, nb, nz, partials, pstride, st);
  return launch_gram_rows<DS, 1, false>(L, w, gb, k, e, nbs, b0, nb, nz, partials, pstride, st);
}

cudaError_t launch_gram_stored(const Layout& L, const void* w1, const int* kb, const double* e, int nbs,
                               int b0, int nb, double* partials, size_t pstride, cudaStream_t st) {
  const int k = *std::max_element(kb, kb + nb);
  if (gram_on_rows(L)) {
    const float* w = reinterpret_cast<const float*>(w1);
    RDM_DISPATCH_DS(L.DS, return (launch_gram_groups<DS>(L, w, k, kb, e, nbs, b0, nb, partials, pstride, st)));
  }
  const int gmax = gram_stored_max_betas(L, k);
  for (int q = 0; q < nb; q += gmax) {
    const int n = std::min(gmax, nb - q);
    double* pq = partials + (size_t)q * pstride;
    RDM_DISPATCH(L, {
      // static reduction scratch (block_reduce_store) + dynamic coefficients: opt in
      const size_t sm = (size_t)k * n * L.groups_per_slice() * DS * DS * sizeof(T) + 16;
      cudaError_t ce = opt_in_smem(reinterpret_cast<const void*>(k_gram_stored<T, DS, VW, 1>));
      if (ce == cudaSuccess) ce = opt_in_smem(reinterpret_cast<const void*>(k_gram_stored<T, DS, VW, 2>));
      if (ce == cudaSuccess)
        ce = opt_in_smem(reinterpret_cast<const void*>(k_gram_stored<T, DS, VW, kGramBetas>));
      if (ce != cudaSuccess) return ce;
      if (n == 1)
        k_gram_stored<T, DS, VW, 1><<<grid_of(L), kThreads, sm, st>>>(
            L, reinterpret_cast<const T*>(w1), k, e, nbs, b0 + q, n, pq, pstride);
      else if (n == 2)
        k_gram_stored<T, DS, VW, 2><<<grid_of(L), kThreads, sm, st>>>(
            L, reinterpret_cast<const T*>(w1), k, e, nbs, b0 + q, n, pq, pstride);
      else
        k_gram_stored<T, DS, VW, kGramBetas><<<grid_of(L), kThreads, sm, st>>>(
            L, reinterpret_cast<const T*>(w1), k, e, nbs, b0 + q, n, pq, pstride);
    });
  }
  return cudaGetLastError();
}

int gram_stored_max_betas(const Layout& L, int k) {
  const size_t per = (size_t)k * L.groups_per_slice() * L.DS * L.DS * L.elem;
  int nb = (int)((160 * 1024) / (per ? per : 1));
  return std::max(0, std::min(nb, kGramBetas));
}

cudaError_t launch_reduce_gram(const Layout& L, const double* partials, size_t pstride, int nb, double* gram,
                               cudaStream_t st) {
  RDM_DISPATCH_DS(L.DS, (k_reduce_gram<DS><<<dim3((unsigned)L.n_groups(), (unsigned)nb), kSmallThreads, 0, st>>>(
                           L, partials, pstride, gram)));
  return cudaGetLastError();
}

// ---------------------------------------------------------------- copy-rate probe
//
// The rate at which TMA bulk copies (the tiled SpMM's only way of filling shared
// memory) move 32 KB chunks from device memory into shared memory: one block per SM,
// one issuing thread, `stages` copies in flight in a ring of shared-memory slots (the
// SpMM's ring depth); the copied data is not read. At step i block b takes chunk
// (i * gridDim.x + b) mod n_chunks: the blocks sweep the buffer together, front to
// back, so a buffer smaller than L2 measures L2 -> shared memory after its first pass
// and a larger one DRAM -> shared memory (no chunk is read twice within a sweep).
// Every wait is
// bounded; a wait that gives up sets *err and the block still waits (bounded) for its
// other copies before it exits.
__global__ void __launch_bounds__(32, 1) k_probe_copy(const unsigned char* src, int64_t n_chunks, int iters,
                                                      int stages, int keep_in_l2, uint32_t* err) {
  extern __shared__ __align__(128) unsigned char smem[];
  uint64_t* const full = reinterpret_cast<uint64_t*>(smem + (size_t)stages * kTileBytes);
  volatile int* const abort_flag = reinterpret_cast<volatile int*>(full + kMaxStages);
  if (threadIdx.x != 0) return;
  for (int i = 0; i < stages; ++i) mbar_init(&full[i], 1);
  *abort_flag = 0;
  fence_mbar_init();
  // normal priority for the L2-resident buffer (it fits anyway; no evict-last lines are
  // left behind for later kernels), evict-first for the streamed one
  uint64_t policy;
  if (keep_in_l2)
    asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;\n" : "=l"(policy));
  else
    policy = policy_evict_first();
  bool ok = true;
  int issued = 0;
  for (int it = 0; it < iters && ok; ++it) {
    const int slot = it % stages;
    if (it >= stages && !ring_wait(&full[slot], (uint32_t)((it / stages - 1) & 1), abort_flag)) {
      ok = false;
      break;
    }
    const int64_t g = ((int64_t)it * gridDim.x + blockIdx.x) % n_chunks;
    mbar_expect_tx(&full[slot], kTileBytes);
    bulk_load_hint(smem + (size_t)slot * kTileBytes, src + (size_t)g * kTileBytes, kTileBytes, &full[slot],
                   policy);
    issued = it + 1;
  }
  // drain: the last min(stages, issued) copies (their slots' most recent phases)
  for (int it = issued > stages ? issued - stages : 0; it < issued; ++it) {
    const int slot = it % stages;
    *abort_flag = 0;
    if (!ring_wait(&full[slot], (uint32_t)((it / stages) & 1), abort_flag)) ok = false;
  }
  if (!ok) atomicOr(err, 1u);
}

cudaError_t launch_probe_copy(const void* src, int64_t n_chunks, int iters, int stages, bool keep_in_l2,
                              uint32_t* err, cudaStream_t st) {
  if (n_chunks <= 0 || iters <= 0 || stages < 1 || stages > kMaxStages) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = opt_in_smem(reinterpret_cast<const void*>(k_probe_copy));
  if (e != cudaSuccess) return e;
  const size_t sm = (size_t)stages * kTileBytes + kMaxStages * 8 + 16;
  k_probe_copy<<<sms, 32, sm, st>>>(static_cast<const unsigned char*>(src), n_chunks, iters, stages,
                                    keep_in_l2 ? 1 : 0, err);
  return cudaGetLastError();
}

}  // namespace rdm
