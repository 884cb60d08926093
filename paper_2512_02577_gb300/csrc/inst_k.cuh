// Launch wrappers for one part of the kernel library -- degree K (PMG_K),
// dimension PMG_DIM, precision PMG_PREC (0 = double, 1 = float) -- and the
// table that exposes them.  inst.cu defines the part's namespace and table
// name from those three macros and includes this file; every wrapper checks
// that the (dim, prec) it is asked for is its own.
#pragma once
#include <cmath>
#include <type_traits>

#include "kernels.cuh"
#include "kernels_def.cuh"
#include "kernels_patch.cuh"

namespace pmg {
namespace PMG_KNS {

constexpr int DP = PMG_DIM;
// the Cartesian patches of this part are solved by the dense sector products
// (K = 1: pointwise) instead of sum factorisation
constexpr bool kDense = K == 1 || PatchDense<DP, TP>::ok() || kStaged;
// the degree's parts of either precision that do so
constexpr bool kProducts64 = PatchDense<DP, double>::ok() || (DP == 3 && (K == 6 || K == 7));
constexpr bool kProducts32 = PatchDense<DP, float>::ok();
// FP64 operator applies by cells; line passes where they are as fast (2D K = 2:
// 9 of a tile's 16 rows used, 0.218 against 0.195 ms at 1024^2 cells) and for
// K = 1 (the 2^d results per cell need more scratch than the passes)
constexpr bool kCellDense = PMG_PREC == 0 && CellDense<DP>::ok() && !(DP == 2 && K == 2);

static int64_t ipow64(int64_t b, int e) { return e == 0 ? 1 : b * ipow64(b, e - 1); }

static bool mine(int dim, int prec) { return dim == DP && prec == PMG_PREC; }

template <int DIM, typename T>
static cudaError_t cart_apply_t(const T* x, T* y, const T* b, T* t0, T* t1, T* t2, T* t3, int n, T s,
                                cudaStream_t st) {
  const int N1 = K * n + 1;
  const int64_t work = (int64_t)(n + 1) * (DIM == 3 ? (int64_t)N1 * N1 : N1);
  const int bs = 256;
  const int g = grid_for(work, bs);
  const FastDiv dnp1(n + 1), dN1(N1);
  if constexpr (DIM == 3 && sizeof(T) == 4) {  // FP32: x and y passes fused per z plane (cart_xy_kernel)
    const int tiles = (n + CartXY<T>::CX - 1) / CartXY<T>::CX;
    cart_xy_kernel<T><<<dim3(tiles, tiles, N1), 256, 0, st>>>(x, t2, t3, n);
    if (b) cart_pass<3, 2, 2, true, T><<<g, bs, 0, st>>>(t2, t3, y, nullptr, b, n, s, dnp1, dN1);
    else cart_pass<3, 2, 2, false, T><<<g, bs, 0, st>>>(t2, t3, y, nullptr, nullptr, n, s, dnp1, dN1);
    g_launches += 2;
    (void)t0;
    (void)t1;
  } else if (DIM == 3) {
    cart_pass<3, 0, 0, false, T><<<g, bs, 0, st>>>(x, nullptr, t0, t1, nullptr, n, s, dnp1, dN1);
    cart_pass<3, 1, 1, false, T><<<g, bs, 0, st>>>(t0, t1, t2, t3, nullptr, n, s, dnp1, dN1);
    if (b) cart_pass<3, 2, 2, true, T><<<g, bs, 0, st>>>(t2, t3, y, nullptr, b, n, s, dnp1, dN1);
    else cart_pass<3, 2, 2, false, T><<<g, bs, 0, st>>>(t2, t3, y, nullptr, nullptr, n, s, dnp1, dN1);
    g_launches += 3;
  } else {
    cart_pass<2, 0, 0, false, T><<<g, bs, 0, st>>>(x, nullptr, t0, t1, nullptr, n, s, dnp1, dN1);
    if (b) cart_pass<2, 1, 2, true, T><<<g, bs, 0, st>>>(t0, t1, y, nullptr, b, n, s, dnp1, dN1);
    else cart_pass<2, 1, 2, false, T><<<g, bs, 0, st>>>(t0, t1, y, nullptr, nullptr, n, s, dnp1, dN1);
    g_launches += 2;
  }
  return cudaGetLastError();
}

static cudaError_t cart_apply(int dim, int prec, const void* x, void* y, const void* b, void* t0, void* t1,
                              void* t2, void* t3, int n, double scale, cudaStream_t s) {
  if (!mine(dim, prec)) return cudaErrorInvalidValue;
  return cart_apply_t<DP, TP>((const TP*)x, (TP*)y, (const TP*)b, (TP*)t0, (TP*)t1, (TP*)t2, (TP*)t3, n, (TP)scale,
                              s);
}

// y = A x or y = b - A x for FP64 vectors in float-float arithmetic
// (cart_pass_ff); t0..t3: FP64-sized scratch, each holding a float-pair plane
template <int DIM>
static cudaError_t cart_apply_ff_t(const double* x, double* y, const double* b, void* t0, void* t1, void* t2,
                                   void* t3, int n, double scale, cudaStream_t st) {
  const int N1 = K * n + 1;
  const int64_t work = (int64_t)(n + 1) * (DIM == 3 ? (int64_t)N1 * N1 : N1);
  const int bs = 256;
  const int g = grid_for(work, bs);
  const FastDiv dnp1(n + 1), dN1(N1);
  const float sh = (float)scale;
  const ff s{sh, (float)(scale - (double)sh)};
  float *f0 = (float*)t0, *f1 = (float*)t1, *f2 = (float*)t2, *f3 = (float*)t3;
  if (DIM == 3) {
    cart_pass_ff<3, 0, 0, false><<<g, bs, 0, st>>>(x, nullptr, f0, f1, nullptr, n, s, dnp1, dN1);
    cart_pass_ff<3, 1, 1, false><<<g, bs, 0, st>>>(f0, f1, f2, f3, nullptr, n, s, dnp1, dN1);
    if (b) cart_pass_ff<3, 2, 2, true><<<g, bs, 0, st>>>(f2, f3, y, nullptr, b, n, s, dnp1, dN1);
    else cart_pass_ff<3, 2, 2, false><<<g, bs, 0, st>>>(f2, f3, y, nullptr, nullptr, n, s, dnp1, dN1);
    g_launches += 3;
  } else {
    cart_pass_ff<2, 0, 0, false><<<g, bs, 0, st>>>(x, nullptr, f0, f1, nullptr, n, s, dnp1, dN1);
    if (b) cart_pass_ff<2, 1, 2, true><<<g, bs, 0, st>>>(f0, f1, y, nullptr, b, n, s, dnp1, dN1);
    else cart_pass_ff<2, 1, 2, false><<<g, bs, 0, st>>>(f0, f1, y, nullptr, nullptr, n, s, dnp1, dN1);
    g_launches += 2;
  }
  return cudaGetLastError();
}

static cudaError_t cart_apply_ff(int dim, const double* x, double* y, const double* b, void* t0, void* t1, void* t2,
                                 void* t3, int n, double scale, cudaStream_t s) {
  if (dim != DP) return cudaErrorInvalidValue;
  return cart_apply_ff_t<DP>(x, y, b, t0, t1, t2, t3, n, scale, s);
}

static int patch_threads(int dim) { return dim == 3 ? PatchShape<3>::TPP : PatchShape<2>::TPP; }

// shared bytes per patch of the patch-major layout
static int patch_smem(int dim, int prec, int n_iter) {
  const int es = prec == 0 ? 8 : 4;
  const int elems = dim == 3 ? (prec == 0 ? PatchShape<3>::stride<double>(n_iter) : PatchShape<3>::stride<float>(n_iter))
                             : (prec == 0 ? PatchShape<2>::stride<double>(n_iter) : PatchShape<2>::stride<float>(n_iter));
  return elems * es;
}

// shared bytes per patch of the interleaved layout (no padding)
static int patch_il_smem(int dim, int prec, int n_iter) {
  const int es = prec == 0 ? 8 : 4;
  const int elems = dim == 3 ? PatchShape<3>::ELEMS + (n_iter > 1 ? 2 * PatchShape<3>::SZT : 0)
                             : PatchShape<2>::ELEMS + (n_iter > 1 ? 2 * PatchShape<2>::SZT : 0);
  return elems * es;
}

static int dinv_len(int dim) {
  int len = 0;
  for (int l = 1; l < nlev(K); ++l) len += ipow(mp(plev(K, l)), dim);
  return len;
}

// shared memory of the block besides its patches: the inverse-diagonal tables
// when the block stages them (stage_dinv)
static int patch_cart_extra_smem(int dim, int prec) {
  const bool staged = dim == 3 ? (prec == 0 ? stage_dinv<3, double>() : stage_dinv<3, float>())
                               : (prec == 0 ? stage_dinv<2, double>() : stage_dinv<2, float>());
  return staged ? dinv_len(dim) * (prec == 0 ? 8 : 4) : 0;
}

// Grid of a persistent patch launch: every block the GPU can hold at once
// (occupancy x SMs), at most one per batch.
static unsigned persistent_grid(const void* kern, int threads, int smem, int64_t nbatch) {
  int dev = 0, sms = 152, per_sm = 1;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const int64_t g = std::min<int64_t>(nbatch, (int64_t)sms * per_sm);
  return (unsigned)std::max<int64_t>(g, 1);
}

// the scale c of a job's results, for FP64 as an integer and an exponent: the
// operands are scaled by 2^(1085 - D - e_window), D the directions in which
// images are summed, and the products by 2^-68
template <int D, typename T>
static void set_scale(DenseJob<T>& J, double c) {
  J.c = (T)c;
  int e = 0;
  const bool finite = std::isfinite(c);
  J.cmul = finite ? (unsigned long long)std::ldexp(std::frexp(c, &e), 64) : 0;
  J.vexp = finite ? e - 64 + 68 - (1085 - D) : 0;
}

template <int DIM, typename T>
static DenseJob<T> dense_job(const T* r, T* dst, int n, const PatchParamsHost& H) {
  DenseJob<T> J{};
  J.r = r;
  J.dst = dst;
  J.table = (const uint4*)H.table;
  J.n = n;
  J.colour = H.colour;
  const double c = (H.colour < 0 ? H.omega_as : 1.0) * (K == 1 ? H.inv_a0 : 1.0 / H.scale);
  set_scale<Sectors<DIM, kPatchM>::SPLIT ? DIM : 0>(J, c);
  J.npatch = (uint32_t)patch_count(DIM, n, H.colour);
  J.d0 = FastDiv(std::max(1, patch_count_1d(n, H.colour, 0)));
  J.d1 = FastDiv(DIM == 3 ? std::max(1, patch_count_1d(n, H.colour, 1)) : 1);
  return J;
}

// patches per block of the dense kernels
template <int DIM, typename T>
constexpr uint32_t dense_batch() { return K == 1 ? 256 : PatchDense<DIM, T>::P; }

// Staged products: the batches of all jobs are numbered job after job, and each
// set of three launches takes the next kStageBatches of them (a job's batches
// in its own stage buffers), so that a group of small levels fills the GPU as
// one large level does.  Solving 16 systems of 4^3 cells together, launches member
// after member and now: K = 6 111 and 17.8 ms, K = 7 248 and 32.7 ms.
template <int DIM>
static cudaError_t stage_launch(const GroupOf<StageJob>& G, cudaStream_t st) {
  using St = Stage<DIM>;
  const unsigned nb = (unsigned)G.start[G.count];
  // while the blocks are less than two per SM, a sector's row tiles in up to
  // three parts of 8, a tile per warp (half cycle, K = 7 at 4^3 cells, sweep: 155 us
  // with one part, 110 with three, 127 by sum factorisation)
  const unsigned z = std::max(1u, std::min((St::MAXT + 7u) / 8u, 304u / (nb * St::S::NS)));
  if (G.count == 1) {
    patch_split_kernel<DIM><<<nb, 256, 0, st>>>(G.job[0]);
    patch_product_kernel<DIM><<<dim3(nb, St::S::NS, z), 256, St::XSM + St::YSM, st>>>(G.job[0]);
    patch_merge_kernel<DIM><<<dim3(nb, St::S::E), 128, St::ZSM, st>>>(G.job[0]);
  } else {
    patch_split_group_kernel<DIM><<<nb, 256, 0, st>>>(G);
    patch_product_group_kernel<DIM><<<dim3(nb, St::S::NS, z), 256, St::XSM + St::YSM, st>>>(G);
    patch_merge_group_kernel<DIM><<<dim3(nb, St::S::E), 128, St::ZSM, st>>>(G);
  }
  g_launches += 3;
  return cudaGetLastError();
}

template <int DIM>
static cudaError_t patch_staged(int count, const PatchSolveJob* jobs, cudaStream_t st) {
  using St = Stage<DIM>;
  GroupOf<StageJob> G;
  G.count = 0;
  G.start[0] = 0;
  cudaError_t e = cudaSuccess;
  for (int j = 0; j < count; ++j) {
    const PatchParamsHost& H = jobs[j].P;
    const int64_t np = patch_count(DIM, jobs[j].n, H.colour), batches = (np + St::P - 1) / St::P;
    if (np == 0) continue;  // no patch (of this colour) on this job's level
    if (np > 0xFFFFFFFFll - 256) return cudaErrorInvalidConfiguration;
    const int64_t room = std::min<int64_t>(H.stage_batches, kStageBatches);
    if (room < 1) return cudaErrorInvalidValue;
    StageJob J;
    J.J = dense_job<DIM, double>((const double*)jobs[j].r, (double*)jobs[j].dst, jobs[j].n, H);
    J.X = (long long*)H.stage;
    J.Y = J.X + H.stage_batches * St::XWORDS;
    J.words = (int*)(J.Y + H.stage_batches * St::YWORDS);
    for (int64_t first = 0; first < batches;) {
      const int64_t nb = std::min({batches - first, room, kStageBatches - G.start[G.count]});
      J.first = (uint32_t)first;
      G.job[G.count] = J;
      G.start[G.count + 1] = G.start[G.count] + nb;
      ++G.count;
      first += nb;
      if (first < batches || G.start[G.count] == kStageBatches) {  // full, or the job needs its buffers again
        if ((e = stage_launch<DIM>(G, st)) != cudaSuccess) return e;
        G.count = 0;
      }
    }
  }
  return G.count > 0 ? stage_launch<DIM>(G, st) : e;
}

template <int DIM, typename T>
static cudaError_t patch_dense_t(const T* r, T* dst, int n, const PatchParamsHost& H, cudaStream_t st) {
  if (patch_count(DIM, n, H.colour) > 0xFFFFFFFFll - 256) return cudaErrorInvalidConfiguration;
  if constexpr (kStaged) {
    const PatchSolveJob job{r, dst, n, H};
    return patch_staged<DIM>(1, &job, st);
  } else {
    const DenseJob<T> J = dense_job<DIM, T>(r, dst, n, H);
    const unsigned grid = (J.npatch + dense_batch<DIM, T>() - 1) / dense_batch<DIM, T>();
    if constexpr (K == 1) patch_point_kernel<DIM, T><<<grid, 256, 0, st>>>(J);
    else patch_dense_kernel<DIM, T><<<grid, 32 * PatchDense<DIM, T>::NW, PatchDense<DIM, T>::SMEM, st>>>(J);
    g_launches += 1;
    return cudaGetLastError();
  }
}

template <int DIM, typename T>
static cudaError_t patch_cart_t(const T* r, T* dst, int n, int ppc, int n_iter, const T* dinv,
                                const PatchParamsHost& H, int* counter, cudaStream_t st) {
  using S = PatchShape<DIM>;
  const int64_t np = patch_count(DIM, n, H.colour);
  if (np == 0) return cudaSuccess;  // no interior vertex (of this colour), no patch
  if constexpr (kDense) return patch_dense_t<DIM, T>(r, dst, n, H, st);
  else {
    if (ppc < 1 || ppc > kMaxPatchesPerBlock) return cudaErrorInvalidValue;
    const int64_t nbatch = (np + ppc - 1) / ppc;
    // more patch lines than threads is fine: every step loops over its lines
    const int threads = std::min(kPatchMaxThreads, (ppc * S::TPP + 31) / 32 * 32);
    const int prec = sizeof(T) == 8 ? 0 : 1;
    const int smem = ppc * patch_smem(DIM, prec, n_iter) + patch_cart_extra_smem(DIM, prec);
    if (smem > kMaxDynSmem) return cudaErrorInvalidConfiguration;
    unsigned grid = (unsigned)nbatch;
    if (counter) {
      grid = persistent_grid((const void*)patch_cart_kernel<DIM, T>, threads, smem, nbatch);
      if (grid < nbatch) {  // more than one wave: persistent blocks
        cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
      } else {
        grid = (unsigned)nbatch;
        counter = nullptr;
      }
    }
    patch_cart_kernel<DIM, T><<<grid, threads, smem, st>>>(r, dst, n, ppc, n_iter, dinv, dinv_len(DIM), to_params<T>(H),
                                                           counter, nbatch);
    g_launches += 1;
    return cudaGetLastError();
  }
}

static cudaError_t patch_cart(int dim, int prec, const void* r, void* dst, int n, int ppc, int n_iter,
                              const void* dinv, const PatchParamsHost& P, int* counter, cudaStream_t s) {
  if (!mine(dim, prec)) return cudaErrorInvalidValue;
  return patch_cart_t<DP, TP>((const TP*)r, (TP*)dst, n, ppc, n_iter, (const TP*)dinv, P, counter, s);
}

// Interleaved layout: patches per block of this part's interleaved kernel
// for n_iter local cycles, or 0 when it has none or they do not fit.
static int patch_il_of(int dim, int prec, int n_iter) {
  if (!mine(dim, prec)) return 0;
  constexpr int il = patch_il<DP, TP>();
  if (il == 0) return 0;
  const int smem = il * patch_il_smem(dim, prec, n_iter) + patch_cart_extra_smem(dim, prec);
  return smem <= kMaxDynSmem ? il : 0;
}

template <int DIM, typename T>
static cudaError_t patch_cart_il_t(const T* r, T* dst, int n, int threads, int n_iter, const T* dinv,
                                   const PatchParamsHost& H, int* counter, cudaStream_t st) {
  const int64_t np = patch_count(DIM, n, H.colour);
  if (np == 0) return cudaSuccess;
  if constexpr (kDense) return patch_dense_t<DIM, T>(r, dst, n, H, st);
  else {
    const int prec = sizeof(T) == 8 ? 0 : 1;
    const int il = patch_il_of(DIM, prec, n_iter);
    if (il == 0 || threads < 32 || threads > 1024 || threads % 32) return cudaErrorInvalidValue;
    const int smem = il * patch_il_smem(DIM, prec, n_iter) + patch_cart_extra_smem(DIM, prec);
    const int64_t nbatch = (np + il - 1) / il;
    unsigned grid = (unsigned)nbatch;
    if (counter) {
      grid = persistent_grid((const void*)patch_cart_il_kernel<DIM, T>, threads, smem, nbatch);
      if (grid < nbatch) {
        cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
      } else {
        grid = (unsigned)nbatch;
        counter = nullptr;
      }
    }
    patch_cart_il_kernel<DIM, T><<<grid, threads, smem, st>>>(r, dst, n, n_iter, dinv, dinv_len(DIM), to_params<T>(H),
                                                              counter, nbatch);
    g_launches += 1;
    return cudaGetLastError();
  }
}

static cudaError_t patch_cart_il(int dim, int prec, const void* r, void* dst, int n, int threads, int n_iter,
                                 const void* dinv, const PatchParamsHost& P, int* counter, cudaStream_t s) {
  if (!mine(dim, prec)) return cudaErrorInvalidValue;
  return patch_cart_il_t<DP, TP>((const TP*)r, (TP*)dst, n, threads, n_iter, (const TP*)dinv, P, counter, s);
}

// u (+)= the summed patch corrections held in dst (add = 0: u = sum)
template <int DIM, typename T>
static cudaError_t patch_gather_t(const T* dst, T* u, int n, int add, cudaStream_t st) {
  const int64_t N = ipow(K * n + 1, DIM);
  if (add) patch_gather_kernel<DIM, true, T><<<grid_for(N, 256), 256, 0, st>>>(dst, u, n, FastDiv(K * n + 1));
  else patch_gather_kernel<DIM, false, T><<<grid_for(N, 256), 256, 0, st>>>(dst, u, n, FastDiv(K * n + 1));
  g_launches += 1;
  return cudaGetLastError();
}

static cudaError_t patch_gather(int dim, int prec, const void* dst, void* u, int n, int add, cudaStream_t s) {
  if (!mine(dim, prec)) return cudaErrorInvalidValue;
  return patch_gather_t<DP, TP>((const TP*)dst, (TP*)u, n, add, s);
}

// one pass of a transfer; ex, ey, ez: extents of its output
template <int AX, bool ADD, typename T>
static void prolong_pass(const T* in, T* out, int nc, int ex, int ey, int ez, cudaStream_t st) {
  hprolong_pass<AX, ADD, T><<<grid_for(transfer_items<AX>(nc, ex, ey, ez), 256), 256, 0, st>>>(
      in, out, nc, ex, ey, ez, FastDiv(ex), FastDiv(ey), FastDiv(nc + 1));
}
template <int AX, typename T>
static void restrict_pass(const T* in, T* out, int nc, int ex, int ey, int ez, cudaStream_t st) {
  hrestrict_pass<AX, T><<<grid_for(transfer_items<AX>(nc, ex, ey, ez), 256), 256, 0, st>>>(
      in, out, nc, ex, ey, ez, FastDiv(ex), FastDiv(ey), FastDiv(nc + 1));
}

template <int DIM, typename T>
static cudaError_t h_prolong_t(const T* uc, T* uf, T* t0, T* t1, int nc, cudaStream_t st) {
  const int c1 = K * nc + 1, f1 = 2 * K * nc + 1;
  if (DIM == 3) {
    prolong_pass<0, false, T>(uc, t0, nc, f1, c1, c1, st);
    prolong_pass<1, false, T>(t0, t1, nc, f1, f1, c1, st);
    prolong_pass<2, true, T>(t1, uf, nc, f1, f1, f1, st);
  } else {
    prolong_pass<0, false, T>(uc, t0, nc, f1, c1, 1, st);
    prolong_pass<1, true, T>(t0, uf, nc, f1, f1, 1, st);
  }
  g_launches += DIM;
  return cudaGetLastError();
}

template <int DIM, typename T>
static cudaError_t h_restrict_t(const T* rf, T* rc, T* t0, T* t1, int nc, cudaStream_t st) {
  const int c1 = K * nc + 1, f1 = 2 * K * nc + 1;
  if (DIM == 3) {
    restrict_pass<2, T>(rf, t0, nc, f1, f1, c1, st);
    restrict_pass<1, T>(t0, t1, nc, f1, c1, c1, st);
    restrict_pass<0, T>(t1, rc, nc, c1, c1, c1, st);
  } else {
    restrict_pass<1, T>(rf, t0, nc, f1, c1, 1, st);
    restrict_pass<0, T>(t0, rc, nc, c1, c1, 1, st);
  }
  g_launches += DIM;
  return cudaGetLastError();
}

static cudaError_t h_prolong_add(int dim, int prec, const void* uc, void* uf, void* t0, void* t1, int nc,
                                 cudaStream_t s) {
  if (!mine(dim, prec)) return cudaErrorInvalidValue;
  return h_prolong_t<DP, TP>((const TP*)uc, (TP*)uf, (TP*)t0, (TP*)t1, nc, s);
}

static cudaError_t h_restrict(int dim, int prec, const void* rf, void* rc, void* t0, void* t1, int nc,
                              cudaStream_t s) {
  if (!mine(dim, prec)) return cudaErrorInvalidValue;
  return h_restrict_t<DP, TP>((const TP*)rf, (TP*)rc, (TP*)t0, (TP*)t1, nc, s);
}

// ---------------------------------------------------------------- grouped launches
// One launch per pass for all jobs; every job's results are those of its own
// launch (each thread takes the same grid-stride slice of every job; the
// patch launch gives each batch of each job to one block).
static int64_t apply_work(int dim, int n) {
  const int64_t N1 = (int64_t)K * n + 1;
  return (int64_t)(n + 1) * (dim == 3 ? N1 * N1 : N1);
}

static bool group_ok(int count) { return count >= 1 && count <= kMaxGroup; }

template <int DIM, typename T>
static cudaError_t cart_apply_group_t(int count, const ApplyJob* jobs, cudaStream_t st) {
  GroupOf<CartPassJob<T>> g0, g1, g2;
  g0.count = g1.count = g2.count = count;
  g0.start[0] = 0;
  int64_t work = 0;
  bool resid = jobs[0].b != nullptr;
  for (int j = 0; j < count; ++j) {
    const ApplyJob& a = jobs[j];
    if ((a.b != nullptr) != resid) return cudaErrorInvalidValue;  // one pass kind per launch
    const T* x = (const T*)a.x;
    T* t0 = (T*)a.t[0];
    T* t1 = (T*)a.t[1];
    T* t2 = (T*)a.t[2];
    T* t3 = (T*)a.t[3];
    const T s = (T)a.scale;
    g0.job[j] = CartPassJob<T>{x, nullptr, t0, t1, nullptr, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
    if (DIM == 3) {
      g1.job[j] = CartPassJob<T>{t0, t1, t2, t3, nullptr, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
      g2.job[j] = CartPassJob<T>{t2, t3, (T*)a.y, nullptr, (const T*)a.b, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
    } else {
      g1.job[j] = CartPassJob<T>{t0, t1, (T*)a.y, nullptr, (const T*)a.b, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
    }
    work += apply_work(DIM, a.n);
    g0.start[j + 1] = work;
  }
  for (int j = 0; j <= count; ++j) g1.start[j] = g2.start[j] = g0.start[j];
  const int bs = 256, g = grid_for(work, bs);
  if (DIM == 3) {
    cart_pass_group<3, 0, 0, false, T><<<g, bs, 0, st>>>(g0);
    cart_pass_group<3, 1, 1, false, T><<<g, bs, 0, st>>>(g1);
    if (resid) cart_pass_group<3, 2, 2, true, T><<<g, bs, 0, st>>>(g2);
    else cart_pass_group<3, 2, 2, false, T><<<g, bs, 0, st>>>(g2);
    g_launches += 3;
  } else {
    cart_pass_group<2, 0, 0, false, T><<<g, bs, 0, st>>>(g0);
    if (resid) cart_pass_group<2, 1, 2, true, T><<<g, bs, 0, st>>>(g1);
    else cart_pass_group<2, 1, 2, false, T><<<g, bs, 0, st>>>(g1);
    g_launches += 2;
  }
  return cudaGetLastError();
}

static cudaError_t cart_apply_group(int dim, int prec, int count, const ApplyJob* jobs, cudaStream_t s) {
  if (!mine(dim, prec) || !group_ok(count)) return cudaErrorInvalidValue;
  return cart_apply_group_t<DP, TP>(count, jobs, s);
}

template <int DIM>
static cudaError_t cart_apply_ff_group_t(int count, const ApplyJob* jobs, cudaStream_t st) {
  GroupOf<CartPassFFJob> g0, g1, g2;
  g0.count = g1.count = g2.count = count;
  g0.start[0] = 0;
  int64_t work = 0;
  const bool resid = jobs[0].b != nullptr;
  for (int j = 0; j < count; ++j) {
    const ApplyJob& a = jobs[j];
    if ((a.b != nullptr) != resid) return cudaErrorInvalidValue;
    const float sh = (float)a.scale;
    const ff s{sh, (float)(a.scale - (double)sh)};
    float *f0 = (float*)a.t[0], *f1 = (float*)a.t[1], *f2 = (float*)a.t[2], *f3 = (float*)a.t[3];
    g0.job[j] = CartPassFFJob{a.x, nullptr, f0, f1, nullptr, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
    if (DIM == 3) {
      g1.job[j] = CartPassFFJob{f0, f1, f2, f3, nullptr, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
      g2.job[j] = CartPassFFJob{f2, f3, a.y, nullptr, (const double*)a.b, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
    } else {
      g1.job[j] = CartPassFFJob{f0, f1, a.y, nullptr, (const double*)a.b, a.n, s, FastDiv(a.n + 1), FastDiv(K * a.n + 1)};
    }
    work += apply_work(DIM, a.n);
    g0.start[j + 1] = work;
  }
  for (int j = 0; j <= count; ++j) g1.start[j] = g2.start[j] = g0.start[j];
  const int bs = 256, g = grid_for(work, bs);
  if (DIM == 3) {
    cart_pass_ff_group<3, 0, 0, false><<<g, bs, 0, st>>>(g0);
    cart_pass_ff_group<3, 1, 1, false><<<g, bs, 0, st>>>(g1);
    if (resid) cart_pass_ff_group<3, 2, 2, true><<<g, bs, 0, st>>>(g2);
    else cart_pass_ff_group<3, 2, 2, false><<<g, bs, 0, st>>>(g2);
    g_launches += 3;
  } else {
    cart_pass_ff_group<2, 0, 0, false><<<g, bs, 0, st>>>(g0);
    if (resid) cart_pass_ff_group<2, 1, 2, true><<<g, bs, 0, st>>>(g1);
    else cart_pass_ff_group<2, 1, 2, false><<<g, bs, 0, st>>>(g1);
    g_launches += 2;
  }
  return cudaGetLastError();
}

static cudaError_t cart_apply_ff_group(int dim, int count, const ApplyJob* jobs, cudaStream_t s) {
  if (dim != DP || !group_ok(count)) return cudaErrorInvalidValue;
  return cart_apply_ff_group_t<DP>(count, jobs, s);
}

template <int DIM, typename T>
static cudaError_t patch_cart_group_t(int count, const PatchSolveJob* jobs, int ppc, int n_iter, const T* dinv,
                                      int* counter, cudaStream_t st) {
  if constexpr (kStaged) {
    return patch_staged<DIM>(count, jobs, st);
  } else if constexpr (kDense) {
    GroupOf<DenseJob<T>> G;
    G.count = 0;
    G.start[0] = 0;
    int64_t grid = 0;
    for (int j = 0; j < count; ++j) {
      const int64_t np = patch_count(DIM, jobs[j].n, jobs[j].P.colour);
      if (np == 0) continue;  // no patch (of this colour) on this job's level
      if (np > 0xFFFFFFFFll - 256) return cudaErrorInvalidConfiguration;
      G.job[G.count++] = dense_job<DIM, T>((const T*)jobs[j].r, (T*)jobs[j].dst, jobs[j].n, jobs[j].P);
      grid += (np + dense_batch<DIM, T>() - 1) / dense_batch<DIM, T>();
      G.start[G.count] = grid;
    }
    if (G.count == 0) return cudaSuccess;
    if (grid > 0x7FFFFFFFll) return cudaErrorInvalidConfiguration;
    if constexpr (K == 1) patch_point_group_kernel<DIM, T><<<(unsigned)grid, 256, 0, st>>>(G);
    else patch_dense_group_kernel<DIM, T><<<(unsigned)grid, 32 * PatchDense<DIM, T>::NW, PatchDense<DIM, T>::SMEM, st>>>(G);
    g_launches += 1;
    return cudaGetLastError();
  } else {
    using S = PatchShape<DIM>;
    if (ppc < 1 || ppc > kMaxPatchesPerBlock) return cudaErrorInvalidValue;
    GroupOf<PatchJob<T>> G;
    G.count = 0;
    G.start[0] = 0;
    int64_t nbatch = 0;
    for (int j = 0; j < count; ++j) {
      const int64_t np = patch_count(DIM, jobs[j].n, jobs[j].P.colour);
      if (np == 0) continue;  // no patch (of this colour) on this job's level
      PatchJob<T>& J = G.job[G.count++];
      J.r = (const T*)jobs[j].r;
      J.dst = (T*)jobs[j].dst;
      J.n = jobs[j].n;
      J.P = to_params<T>(jobs[j].P);
      nbatch += (np + ppc - 1) / ppc;
      G.start[G.count] = nbatch;
    }
    if (G.count == 0) return cudaSuccess;
    const int threads = std::min(kPatchMaxThreads, (ppc * S::TPP + 31) / 32 * 32);
    const int prec = sizeof(T) == 8 ? 0 : 1;
    const int smem = ppc * patch_smem(DIM, prec, n_iter) + patch_cart_extra_smem(DIM, prec);
    if (smem > kMaxDynSmem) return cudaErrorInvalidConfiguration;
    unsigned grid = (unsigned)nbatch;
    if (counter) {
      grid = persistent_grid((const void*)patch_cart_group_kernel<DIM, T>, threads, smem, nbatch);
      if (grid < nbatch) {
        cudaError_t e = cudaMemsetAsync(counter, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
      } else {
        grid = (unsigned)nbatch;
        counter = nullptr;
      }
    }
    patch_cart_group_kernel<DIM, T><<<grid, threads, smem, st>>>(ppc, n_iter, dinv, dinv_len(DIM), counter, nbatch, G);
    g_launches += 1;
    return cudaGetLastError();
  }
}

// ---------------------------------------------------------------- dense patch operator
// Device bytes of the part's table of sector matrices (0: not a dense part)
// and of the FP64 scratch that its set-up needs: the columns' low parts and
// the exponents of orbits and rows.  The columns themselves end the table.
static int64_t patch_table_bytes(int dim, int prec) {
  if (!mine(dim, prec) || !kDense || K == 1) return 0;
  return PatchDense<DP, TP>::TABLE_BYTES;
}

template <class S>
constexpr int64_t sector_scratch_bytes() {
  return 8 * (int64_t)S::ORBITS * S::NODES + 4 * (S::ORBITS + S::ROWS);
}
template <class S>
static int* sector_exponents(double* scratch) { return (int*)(scratch + (int64_t)S::ORBITS * S::NODES); }

static int64_t patch_scratch_bytes(int dim) { return dim == DP ? sector_scratch_bytes<Sectors<DP, kPatchM>>() : 0; }

static double* patch_columns(int dim, int prec, void* table) {
  return mine(dim, prec) ? (double*)((char*)table + PatchDense<DP, TP>::COLUMNS) : nullptr;
}

template <int DIM, typename V>
static cudaError_t patch_columns_t(const PatchParamsHost& H, int n_iter, const double* dinv, double* columns,
                                   double* scratch, cudaStream_t st) {
  using S = Sectors<DIM, kPatchM>;
  const int np = std::max(1, 32 / PatchShape<DIM>::TPP);  // few: a block's FP64 work is its latency
  const int threads = std::min(256, (np * PatchShape<DIM>::TPP + 31) / 32 * 32);
  const int smem = np * PatchShape<DIM>::ELEMS * (int)sizeof(V);
  if (smem > kMaxDynSmem) return cudaErrorInvalidConfiguration;
  for (int it = 0; it < n_iter; ++it)
    patch_columns_kernel<DIM, V><<<(S::ORBITS + np - 1) / np, threads, smem, st>>>(
        columns, scratch, sector_exponents<S>(scratch), np, it == 0, dinv, to_params<double>(H));
  g_launches += n_iter;
  return cudaGetLastError();
}

// exponents of the sector matrices from the columns: the orbits', then the rows'
template <int DIM, int M>
static cudaError_t sector_exponents_t(const double* columns, double* scratch, cudaStream_t st) {
  using S = Sectors<DIM, M>;
  int* exps = sector_exponents<S>(scratch);
  sector_exponents_kernel<DIM, M><<<(S::ROWS + 3) / 4, 128, 0, st>>>(columns, exps + S::ORBITS, exps);
  g_launches += 1;
  return cudaGetLastError();
}

// fragments (and FP64 exponents) of a table from its columns and the scratch
template <int DIM, typename T, int M>
static cudaError_t sector_table_t(const double* columns, double* scratch, void* table, cudaStream_t st) {
  using S = Sectors<DIM, M>;
  const int* exps = sector_exponents<S>(scratch);
  sector_table_kernel<DIM, T, M><<<(S::TILES * 128 + 255) / 256, 256, 0, st>>>(columns, scratch, exps + S::ORBITS, exps,
                                                                               (uint32_t*)table);
  g_launches += 1;
  return cudaGetLastError();
}

// FP64 part: columns of the local solver (unit scale; dinv: its inverse
// diagonals) for products in precision prec, and the exponents
template <int DIM, typename T>
static cudaError_t patch_entries_t(const PatchParamsHost& H, int n_iter, bool fp64, const double* dinv,
                                   double* columns, double* scratch, cudaStream_t st) {
  if constexpr (sizeof(T) == 8 && K > 1) {
    cudaError_t e = cudaErrorInvalidValue;  // no such product part
    if (fp64) {
      if constexpr (kProducts64) {
        e = patch_columns_t<DIM, dd>(H, n_iter, dinv, columns, scratch, st);
        if (e == cudaSuccess) e = sector_exponents_t<DIM, kPatchM>(columns, scratch, st);
      }
    } else {
      if constexpr (kProducts32) e = patch_columns_t<DIM, double>(H, n_iter, dinv, columns, scratch, st);
    }
    return e;
  }
  return cudaErrorInvalidValue;
}

static cudaError_t patch_entries(int dim, const PatchParamsHost& H, int n_iter, int prec, const double* dinv,
                                 double* columns, double* scratch, cudaStream_t st) {
  if (dim != DP) return cudaErrorInvalidValue;
  return patch_entries_t<DP, TP>(H, n_iter, prec == 0, dinv, columns, scratch, st);
}

// the part's table from its columns and the scratch
template <int DIM, typename T>
static cudaError_t patch_table_t(double* scratch, void* table, cudaStream_t st) {
  if constexpr (kDense && K > 1)
    return sector_table_t<DIM, T, kPatchM>(patch_columns(DIM, sizeof(T) == 8 ? 0 : 1, table), scratch, table, st);
  return cudaErrorInvalidValue;
}

// bytes of the stage buffers for `batches` batches of patches, and the batches
// they are to hold for a level of n cells (0: not a staged part)
template <int DIM>
static int64_t stage_bytes_t(int64_t batches) {
  if constexpr (kStaged) return batches * Stage<DIM>::BYTES;
  return 0;
}
template <int DIM>
static int64_t stage_batches_t(int n) {
  if constexpr (kStaged)
    return std::min<int64_t>(kStageBatches, (patch_count(DIM, n, -1) + Stage<DIM>::P - 1) / Stage<DIM>::P);
  return 0;
}
static int64_t patch_stage_bytes(int64_t batches) { return stage_bytes_t<DP>(batches); }
static int64_t patch_stage_batches(int n) { return stage_batches_t<DP>(n); }

// ---------------------------------------------------------------- FP64 apply by cells
static int64_t cell_table_bytes(int dim) { return dim == DP && kCellDense ? CellDense<DP>::TABLE_BYTES : 0; }
static int64_t cell_scratch_bytes(int dim) {
  return dim == DP && kCellDense ? sector_scratch_bytes<Sectors<DP, kCellM>>() : 0;
}

// the cell's table, by way of the scratch (used on the stream, free again afterwards)
template <int DIM, typename T>
static cudaError_t cell_table_t(double* scratch, void* table, cudaStream_t st) {
  if constexpr (kCellDense) {
    using S = Sectors<DIM, kCellM>;
    double* columns = (double*)((char*)table + CellDense<DIM>::COLUMNS);
    cell_columns_kernel<DIM><<<(S::ORBITS * S::NODES + 255) / 256, 256, 0, st>>>(columns, scratch,
                                                                               sector_exponents<S>(scratch));
    g_launches += 1;
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess) e = sector_exponents_t<DIM, kCellM>(columns, scratch, st);
    if (e == cudaSuccess) e = sector_table_t<DIM, double, kCellM>(columns, scratch, table, st);
    return e;
  }
  return cudaErrorInvalidValue;
}

static cudaError_t cell_table(int dim, double* scratch, void* table, cudaStream_t st) {
  if (dim != DP) return cudaErrorInvalidValue;
  return cell_table_t<DP, TP>(scratch, table, st);
}

// the cells of a level; cells: n^d (K+1)^d doubles of scratch
template <int DIM>
static DenseJob<double> cell_job(const double* x, double* cells, const void* table, int n, double scale) {
  DenseJob<double> J{};
  J.r = x;
  J.dst = cells;
  J.table = (const uint4*)table;
  J.n = n;
  J.colour = -1;
  set_scale<Sectors<DIM, kCellM>::SPLIT ? DIM : 0>(J, scale);
  J.npatch = (uint32_t)ipow64(n, DIM);
  J.d0 = FastDiv(n);
  J.d1 = FastDiv(DIM == 3 ? n : 1);
  return J;
}

// Levels whose cells are multiplied; on the others the line passes are faster:
// up to 8^3 cells of K = 8 (32 blocks, one per SM for its 216 KB, 62-67 us; 57-58
// us by lines; at 12^3 81 and 187)
template <int DIM>
static bool cells_pay(int n) { return !(DIM == 3 && K == 8) || n > 8; }

// t: scratch of cart_apply; t[0] also holds n^d (K+1)^d doubles
template <int DIM, typename T>
static cudaError_t cell_apply_t(const double* x, double* y, const double* b, double* const* t, const void* table, int n,
                                double scale, cudaStream_t st) {
  if constexpr (kCellDense) {
    if (!cells_pay<DIM>(n)) return cart_apply_t<DIM, double>(x, y, b, t[0], t[1], t[2], t[3], n, scale, st);
    using D = CellDense<DIM>;
    double* cells = t[0];
    const DenseJob<double> J = cell_job<DIM>(x, cells, table, n, scale);
    cell_dense_kernel<DIM><<<(J.npatch + D::P - 1) / D::P, 32 * D::NW, D::SMEM, st>>>(J);
    const int64_t N = ipow64(K * n + 1, DIM);
    cell_sum_kernel<DIM><<<(unsigned)((N + 255) / 256), 256, 0, st>>>(CellSumJob<DIM>{cells, b, y, n, FastDiv(K * n + 1)}, N);
    g_launches += 2;
    return cudaGetLastError();
  }
  return cudaErrorInvalidValue;
}

static cudaError_t cell_apply(int dim, const double* x, double* y, const double* b, double* const* t, const void* table,
                              int n, double scale, cudaStream_t st) {
  if (dim != DP) return cudaErrorInvalidValue;
  return cell_apply_t<DP, TP>(x, y, b, t, table, n, scale, st);
}

template <int DIM, typename T>
static cudaError_t cell_apply_group_t(int count, const ApplyJob* jobs, cudaStream_t st) {
  if constexpr (kCellDense) {
    using D = CellDense<DIM>;
    GroupOf<DenseJob<double>> G;
    GroupOf<CellSumJob<DIM>> H;
    G.start[0] = H.start[0] = 0;
    ApplyJob lines[kMaxGroup];  // the members whose level takes the line passes
    int m = 0, nl = 0;
    for (int i = 0; i < count; ++i) {
      const ApplyJob& a = jobs[i];
      if (!cells_pay<DIM>(a.n)) {
        lines[nl++] = a;
        continue;
      }
      G.job[m] = cell_job<DIM>((const double*)a.x, (double*)a.t[0], a.table, a.n, a.scale);
      G.start[m + 1] = G.start[m] + (G.job[m].npatch + D::P - 1) / D::P;
      H.job[m] = CellSumJob<DIM>{(const double*)a.t[0], (const double*)a.b, (double*)a.y, a.n, FastDiv(K * a.n + 1)};
      H.start[m + 1] = H.start[m] + ipow64(K * a.n + 1, DIM);
      ++m;
    }
    G.count = H.count = m;
    if (nl > 0) {
      cudaError_t e = cart_apply_group_t<DIM, double>(nl, lines, st);
      if (e != cudaSuccess || m == 0) return e;
    }
    cell_dense_group_kernel<DIM><<<(unsigned)G.start[m], 32 * D::NW, D::SMEM, st>>>(G);
    cell_sum_group_kernel<DIM><<<(unsigned)((H.start[m] + 255) / 256), 256, 0, st>>>(H);
    g_launches += 2;
    return cudaGetLastError();
  }
  return cudaErrorInvalidValue;
}

static cudaError_t cell_apply_group(int dim, int count, const ApplyJob* jobs, cudaStream_t st) {
  if (dim != DP || !group_ok(count)) return cudaErrorInvalidValue;
  return cell_apply_group_t<DP, TP>(count, jobs, st);
}

static cudaError_t patch_table(int dim, int prec, double* scratch, void* table, cudaStream_t st) {
  if (!mine(dim, prec)) return cudaErrorInvalidValue;
  return patch_table_t<DP, TP>(scratch, table, st);
}

static cudaError_t patch_cart_group(int dim, int prec, int count, const PatchSolveJob* jobs, int ppc, int n_iter,
                                    const void* dinv, int* counter, cudaStream_t s) {
  if (!mine(dim, prec) || !group_ok(count)) return cudaErrorInvalidValue;
  return patch_cart_group_t<DP, TP>(count, jobs, ppc, n_iter, (const TP*)dinv, counter, s);
}

template <int DIM, typename T>
static cudaError_t patch_gather_group_t(int count, const GatherSolveJob* jobs, int add, cudaStream_t st) {
  GroupOf<GatherJob<T>> G;
  G.count = count;
  G.start[0] = 0;
  int64_t work = 0;
  for (int j = 0; j < count; ++j) {
    G.job[j] = GatherJob<T>{(const T*)jobs[j].dst, (T*)jobs[j].u, jobs[j].n, FastDiv(K * jobs[j].n + 1)};
    work += ipow(K * jobs[j].n + 1, DIM);
    G.start[j + 1] = work;
  }
  if (add) patch_gather_group<DIM, true, T><<<grid_for(work, 256), 256, 0, st>>>(G);
  else patch_gather_group<DIM, false, T><<<grid_for(work, 256), 256, 0, st>>>(G);
  g_launches += 1;
  return cudaGetLastError();
}

static cudaError_t patch_gather_group(int dim, int prec, int count, const GatherSolveJob* jobs, int add,
                                     cudaStream_t s) {
  if (!mine(dim, prec) || !group_ok(count)) return cudaErrorInvalidValue;
  return patch_gather_group_t<DP, TP>(count, jobs, add, s);
}

// The passes of h_prolong_t / h_restrict_t with each job's extents.
template <typename T>
static TransferJob<T> transfer_job(const T* in, T* out, int nc, int ex, int ey, int ez) {
  return TransferJob<T>{in, out, nc, ex, ey, ez, FastDiv(ex), FastDiv(ey), FastDiv(nc + 1)};
}

template <int DIM, typename T>
static cudaError_t h_prolong_group_t(int count, const TransferSolveJob* jobs, cudaStream_t st) {
  GroupOf<TransferJob<T>> g[3];
  int64_t work[3] = {0, 0, 0};
  for (int i = 0; i < 3; ++i) {
    g[i].count = count;
    g[i].start[0] = 0;
  }
  for (int j = 0; j < count; ++j) {
    const TransferSolveJob& a = jobs[j];
    const int nc = a.nc, c1 = K * nc + 1, f1 = 2 * K * nc + 1;
    const T* uc = (const T*)a.in;
    T *uf = (T*)a.out, *t0 = (T*)a.t0, *t1 = (T*)a.t1;
    if (DIM == 3) {
      g[0].job[j] = transfer_job<T>(uc, t0, nc, f1, c1, c1);
      g[1].job[j] = transfer_job<T>(t0, t1, nc, f1, f1, c1);
      g[2].job[j] = transfer_job<T>(t1, uf, nc, f1, f1, f1);
      work[0] += transfer_items<0>(nc, f1, c1, c1);
      work[1] += transfer_items<1>(nc, f1, f1, c1);
      work[2] += transfer_items<2>(nc, f1, f1, f1);
    } else {
      g[0].job[j] = transfer_job<T>(uc, t0, nc, f1, c1, 1);
      g[1].job[j] = transfer_job<T>(t0, uf, nc, f1, f1, 1);
      work[0] += transfer_items<0>(nc, f1, c1, 1);
      work[1] += transfer_items<1>(nc, f1, f1, 1);
    }
    for (int i = 0; i < 3; ++i) g[i].start[j + 1] = work[i];
  }
  const int bs = 256;
  if (DIM == 3) {
    hprolong_group<0, false, T><<<grid_for(work[0], bs), bs, 0, st>>>(g[0]);
    hprolong_group<1, false, T><<<grid_for(work[1], bs), bs, 0, st>>>(g[1]);
    hprolong_group<2, true, T><<<grid_for(work[2], bs), bs, 0, st>>>(g[2]);
    g_launches += 3;
  } else {
    hprolong_group<0, false, T><<<grid_for(work[0], bs), bs, 0, st>>>(g[0]);
    hprolong_group<1, true, T><<<grid_for(work[1], bs), bs, 0, st>>>(g[1]);
    g_launches += 2;
  }
  return cudaGetLastError();
}

template <int DIM, typename T>
static cudaError_t h_restrict_group_t(int count, const TransferSolveJob* jobs, cudaStream_t st) {
  GroupOf<TransferJob<T>> g[3];
  int64_t work[3] = {0, 0, 0};
  for (int i = 0; i < 3; ++i) {
    g[i].count = count;
    g[i].start[0] = 0;
  }
  for (int j = 0; j < count; ++j) {
    const TransferSolveJob& a = jobs[j];
    const int nc = a.nc, c1 = K * nc + 1, f1 = 2 * K * nc + 1;
    const T* rf = (const T*)a.in;
    T *rc = (T*)a.out, *t0 = (T*)a.t0, *t1 = (T*)a.t1;
    if (DIM == 3) {
      g[0].job[j] = transfer_job<T>(rf, t0, nc, f1, f1, c1);
      g[1].job[j] = transfer_job<T>(t0, t1, nc, f1, c1, c1);
      g[2].job[j] = transfer_job<T>(t1, rc, nc, c1, c1, c1);
      work[0] += transfer_items<2>(nc, f1, f1, c1);
      work[1] += transfer_items<1>(nc, f1, c1, c1);
      work[2] += transfer_items<0>(nc, c1, c1, c1);
    } else {
      g[0].job[j] = transfer_job<T>(rf, t0, nc, f1, c1, 1);
      g[1].job[j] = transfer_job<T>(t0, rc, nc, c1, c1, 1);
      work[0] += transfer_items<1>(nc, f1, c1, 1);
      work[1] += transfer_items<0>(nc, c1, c1, 1);
    }
    for (int i = 0; i < 3; ++i) g[i].start[j + 1] = work[i];
  }
  const int bs = 256;
  if (DIM == 3) {
    hrestrict_group<2, T><<<grid_for(work[0], bs), bs, 0, st>>>(g[0]);
    hrestrict_group<1, T><<<grid_for(work[1], bs), bs, 0, st>>>(g[1]);
    hrestrict_group<0, T><<<grid_for(work[2], bs), bs, 0, st>>>(g[2]);
    g_launches += 3;
  } else {
    hrestrict_group<1, T><<<grid_for(work[0], bs), bs, 0, st>>>(g[0]);
    hrestrict_group<0, T><<<grid_for(work[1], bs), bs, 0, st>>>(g[1]);
    g_launches += 2;
  }
  return cudaGetLastError();
}

static cudaError_t h_prolong_add_group(int dim, int prec, int count, const TransferSolveJob* jobs, cudaStream_t s) {
  if (!mine(dim, prec) || !group_ok(count)) return cudaErrorInvalidValue;
  return h_prolong_group_t<DP, TP>(count, jobs, s);
}

static cudaError_t h_restrict_group(int dim, int prec, int count, const TransferSolveJob* jobs, cudaStream_t s) {
  if (!mine(dim, prec) || !group_ok(count)) return cudaErrorInvalidValue;
  return h_restrict_group_t<DP, TP>(count, jobs, s);
}

// Opt every kernel of this degree into the largest dynamic shared memory the
// device allows next to the kernel's static shared memory (called once per
// device at context creation, outside any stream capture).
template <class Kern>
static cudaError_t allow_smem(Kern k, int optin) {
  cudaFuncAttributes a;
  cudaError_t e = cudaFuncGetAttributes(&a, k);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)a.sharedSizeBytes);
  if (e != cudaSuccess) return e;
  // prefer the largest shared-memory carve-out: these kernels live in it
  return cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
}

static int max_threads_of(const void* k) {
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, k) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return a.maxThreadsPerBlock;
}

template <int DIM, typename T>
static int cart_max_threads(bool interleaved) {
  if constexpr (kDense) return !interleaved ? kPatchMaxThreads : (sizeof(T) == 8 ? 768 : 1024);  // no effect
  else if (!interleaved) return max_threads_of((const void*)patch_cart_kernel<DIM, T>);
  else return max_threads_of((const void*)patch_cart_il_kernel<DIM, T>);
}

static int patch_max_threads(int dim, int prec, int deformed) {
  if (!mine(dim, prec)) return 0;
  if (deformed)
    return std::min(max_threads_of((const void*)patch_def_kernel<DP, TP, float>),
                    max_threads_of((const void*)patch_def_kernel<DP, TP, double>));
  return cart_max_threads<DP, TP>(false);
}

static int patch_il_max_threads(int dim, int prec) {
  if (!mine(dim, prec) || patch_il<DP, TP>() == 0) return 0;
  return cart_max_threads<DP, TP>(true);
}

template <int DIM, typename T, class Acc>
static void prepare_cart(int optin, const Acc& acc) {
  if constexpr (!kDense) {
    acc(allow_smem(patch_cart_kernel<DIM, T>, optin));
    acc(allow_smem(patch_cart_group_kernel<DIM, T>, optin));
    if (patch_il<DIM, T>() > 0) acc(allow_smem(patch_cart_il_kernel<DIM, T>, optin));
  } else if constexpr (kStaged) {
    acc(allow_smem(patch_product_kernel<DIM>, optin));
    acc(allow_smem(patch_product_group_kernel<DIM>, optin));
    acc(allow_smem(patch_merge_kernel<DIM>, optin));
    acc(allow_smem(patch_merge_group_kernel<DIM>, optin));
  } else if constexpr (K > 1) {
    acc(allow_smem(patch_dense_kernel<DIM, T>, optin));
    acc(allow_smem(patch_dense_group_kernel<DIM, T>, optin));
  }
  if constexpr (kCellDense) {
    acc(allow_smem(cell_dense_kernel<DIM>, optin));
    acc(allow_smem(cell_dense_group_kernel<DIM>, optin));
  }
  if constexpr (sizeof(T) == 8 && K > 1) {
    if constexpr (kProducts32) acc(allow_smem(patch_columns_kernel<DIM, double>, optin));
    if constexpr (kProducts64) acc(allow_smem(patch_columns_kernel<DIM, dd>, optin));
  }
}

static cudaError_t prepare() {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  cudaError_t r = cudaSuccess;
  auto acc = [&](cudaError_t x) { if (x != cudaSuccess && r == cudaSuccess) r = x; };
  prepare_cart<DP, TP>(optin, acc);
  acc(allow_smem(patch_def_kernel<DP, TP, float>, optin));
  acc(allow_smem(patch_def_kernel<DP, TP, double>, optin));
  acc(allow_smem(def_cell_kernel<DP, TP, float>, optin));
  acc(allow_smem(def_cell_kernel<DP, TP, double>, optin));
  return r;
}

}  // namespace PMG_KNS

const KernelTable* PMG_TABLE_FN() {
  static KernelTable t = {
      PMG_K,
      PMG_DIM,
      PMG_PREC,
      PMG_KNS::prepare,
      PMG_KNS::cart_apply,
      PMG_KNS::patch_cart,
      PMG_KNS::patch_gather,
      PMG_KNS::patch_cart_extra_smem,
      PMG_KNS::patch_threads,
      PMG_KNS::patch_smem,
      PMG_KNS::h_prolong_add,
      PMG_KNS::h_restrict,
      PMG_KNS::def_apply,
      PMG_KNS::patch_def,
      PMG_KNS::patch_def_threads,
      PMG_KNS::patch_def_smem,
      PMG_KNS::patch_max_threads,
      PMG_KNS::patch_il_of,
      PMG_KNS::patch_cart_il,
      PMG_KNS::patch_il_max_threads,
      PMG_KNS::cart_apply_ff,
      PMG_KNS::def_apply_ff,
      PMG_KNS::def_apply_candidates,
      PMG_KNS::cart_apply_group,
      PMG_KNS::cart_apply_ff_group,
      PMG_KNS::patch_cart_group,
      PMG_KNS::patch_gather_group,
      PMG_KNS::h_prolong_add_group,
      PMG_KNS::h_restrict_group,
      PMG_KNS::patch_table_bytes,
      PMG_KNS::patch_scratch_bytes,
      PMG_KNS::patch_columns,
      PMG_KNS::patch_entries,
      PMG_KNS::patch_table,
      PMG_KNS::patch_stage_bytes,
      PMG_KNS::patch_stage_batches,
      PMG_KNS::cell_table_bytes,
      PMG_KNS::cell_scratch_bytes,
      PMG_KNS::cell_table,
      PMG_KNS::cell_apply,
      PMG_KNS::cell_apply_group,
  };
  return &t;
}

}  // namespace pmg
