// Host-side launchers of the step kernels, one KernelSet per (dimension,
// degree, equation, precision).  The host context only sees KernelSet.
#pragma once
#include "cr_kernels.cuh"

namespace crk {

struct KernelSet {
  int dim, degree, nvars, nodes, mixed;
  int launches_per_step;
  // params points at a KParams<double> (FP64) or KParams<float> (FP32_BULK)
  cudaError_t (*step)(const void* params, cudaStream_t s);
  cudaError_t (*launch[4])(const void* params, cudaStream_t s);  // local, face, update, finish
  const char* names[4];
  cudaError_t (*prologue)(const void* params, cudaStream_t s);
  cudaError_t (*split)(const void* params, const double* in, cudaStream_t s);  // FP64 -> state
  cudaError_t (*join)(const void* params, double* out, cudaStream_t s);        // state -> FP64
  cudaError_t (*means)(const void* params, double* out, cudaStream_t s);       // [M][Ne] FP64
  cudaError_t (*configure)();
};

template <int DIM, int N, class EQ, typename real, bool MIXED>
struct Impl {
  static constexpr int n = N + 1;
  static constexpr int NP = DIM == 2 ? n * n : n;
  static constexpr int M = EQ::M;
  static constexpr int NFN = DIM == 2 ? n : 1;
  using LB = LocalBlocks<DIM, N, EQ, MIXED>;
  // variables per node in the element kernel's shared arrays (VarPack pads FP32 to pairs)
  static constexpr int MV = (M + VarPack<real>::VL - 1) / VarPack<real>::VL * VarPack<real>::VL;

  // elements of a 256-thread block (at least one); the FP32-bulk update kernel
  // takes UpdateShape's (128 threads), small 1D meshes kSmallThreads
  static constexpr int EPB = BlockShape<NP>::EPB;

  static size_t smem_local(int epb) {
    if constexpr (HasLocal64<DIM, EQ, MIXED>::value)
      return (size_t)5 * M * epb * NP * sizeof(double) + local64_extra<DIM, N, EQ>(epb);
    return (((size_t)5 * MV * epb * NP * sizeof(real) + 15) & ~(size_t)15) + (size_t)epb * sizeof(double) +
           (size_t)4 * n * n * sizeof(real) + (size_t)epb * 4 * sizeof(int);
  }
  static constexpr int RW = 2 * M > 4 ? 2 * M : 4;
  static constexpr int MU = M > 2 ? M : 2;
  static size_t smem_update(int epb) {
    return ((size_t)(MU + RW) * epb * NP + 16 * (size_t)epb) * sizeof(double) +
           (size_t)epb * (NP + 1) * sizeof(float);
  }

  static cudaError_t configure() {
    cudaError_t err;
    err = cudaFuncSetAttribute(k_local<DIM, N, EQ, real, MIXED>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_local(EPB));
    if (err != cudaSuccess) return err;
    if constexpr (LB::many > LB::value) {
      err = cudaFuncSetAttribute(k_local<DIM, N, EQ, real, MIXED, 256, LB::many>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_local(EPB));
      if (err != cudaSuccess) return err;
    }
    err = cudaFuncSetAttribute(k_update<DIM, N, EQ, real, MIXED>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_update(EPB));
    if (err != cudaSuccess) return err;
    return cudaFuncSetAttribute(k_prologue<DIM, N, EQ, real, MIXED>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_update(EPB));
  }

  static int sm_count() {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 152;
    return n;
  }

  // One-dimensional FP64 meshes whose blocks of kSmallThreads threads are all resident
  // at once take those (the kernels are bound by the FP64 pipe of the SMs that have
  // work, and 256-thread blocks leave SMs idle); past that a second wave begins, where
  // 256-thread blocks may still fit.  us per step with 64 and 256 threads, 152 SMs: 1D
  // Euler N = 4 (72,960 nodes at once), 10,000 nodes 63 and 68, 60,000 72 and 75, 77,000 93
  // and 71, 120,000 100 and 102; N = 2 (76,608) 60,000 62 and 64, 77,000 72 and 60; linear
  // advection N = 3, 40,000 27 and 29.  FP32 bulk is latency bound: the same within 1%.
  static constexpr bool kHasSmall = DIM == 1 && !MIXED;
  static constexpr int kSmallThreads = 64;
  static bool small(const KParams<real>& P) {
    constexpr int E = BlockShape<NP, kSmallThreads>::EPB;
    return kHasSmall && (P.m.ne + E - 1) / E <= sm_count() * LB::value * (256 / kSmallThreads);
  }

  // Launch behind the previous kernel of the step (wait_for_previous_kernel).
  template <class... A>
  static cudaError_t chain(void (*kernel)(A...), int grid, int threads, size_t smem, cudaStream_t s, const A&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...);
  }

  template <int THREADS>
  static cudaError_t local_in(const KParams<real>& P, cudaStream_t s) {
    constexpr int E = BlockShape<NP, THREADS>::EPB;
    const int blocks = (P.m.ne + E - 1) / E;
    if constexpr (LB::many > LB::value)  // more blocks than are resident at once: one more per SM
      if (blocks > sm_count() * LB::value)
        return chain(&k_local<DIM, N, EQ, real, MIXED, THREADS, LB::many>, blocks, E * NP, smem_local(E), s, P);
    return chain(&k_local<DIM, N, EQ, real, MIXED, THREADS>, blocks, E * NP, smem_local(E), s, P);
  }
  template <int THREADS>
  static cudaError_t update_in(const KParams<real>& P, cudaStream_t s) {
    constexpr int E = UpdateShape<NP, MIXED, THREADS>::EPB;
    return chain(&k_update<DIM, N, EQ, real, MIXED, THREADS>, (P.m.ne + E - 1) / E, E * NP, smem_update(E), s, P);
  }
  static cudaError_t launch_local(const void* pv, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    if constexpr (kHasSmall)
      if (small(P)) return local_in<kSmallThreads>(P, s);
    return local_in<256>(P, s);
  }
  static cudaError_t launch_face(const void* pv, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    const int nfaces = P.m.ny * P.m.nfx * NFN + (DIM == 2 ? P.m.nfy * P.m.nx * n : 0);
    // few face nodes: one warp per block, so that every SM has some
    const int threads = nfaces < sm_count() * 4 * 32 ? 32 : 256;
    return chain(&k_face<DIM, N, EQ, real>, (nfaces + threads - 1) / threads, threads, 0, s, P);
  }
  static cudaError_t launch_update(const void* pv, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    if constexpr (kHasSmall)
      if (small(P)) return update_in<kSmallThreads>(P, s);
    return update_in<256>(P, s);
  }
  static cudaError_t launch_finish(const void* pv, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    return chain(&k_finish_step, 1, 32, 0, s, P.b.ctl);
  }
  static cudaError_t step(const void* pv, cudaStream_t s) {
    cudaError_t e = launch_local(pv, s);
    if (e == cudaSuccess) e = launch_face(pv, s);
    if (e == cudaSuccess) e = launch_update(pv, s);
    if (e == cudaSuccess) e = launch_finish(pv, s);
    return e;
  }

  static cudaError_t prologue(const void* pv, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    const int E = small(P) ? BlockShape<NP, kSmallThreads>::EPB : EPB;
    k_prologue<DIM, N, EQ, real, MIXED><<<(P.m.ne + E - 1) / E, E * NP, smem_update(E), s>>>(P);
    return cudaGetLastError();
  }

  static cudaError_t split(const void* pv, const double* in, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    const size_t nvals = (size_t)M * P.m.ne * NP;
    if constexpr (MIXED) {
      const int nthr = M * P.m.ne;
      k_split_state<DIM, N, M><<<(nthr + kRowsPerBlock - 1) / kRowsPerBlock, kRowsPerBlock, 0, s>>>(
          in, P.b.u, P.b.umean, P.b.umean_f, P.m.ne, P.td);
      return cudaGetLastError();
    } else {
      return cudaMemcpyAsync(P.b.u, in, nvals * sizeof(double), cudaMemcpyDefault, s);
    }
  }

  static cudaError_t join(const void* pv, double* out, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    const size_t nvals = (size_t)M * P.m.ne * NP;
    if constexpr (MIXED) {
      k_join_state<NP><<<(int)((nvals + 255) / 256), 256, 0, s>>>(P.b.u, P.b.umean, out, (int)nvals);
      return cudaGetLastError();
    } else {
      return cudaMemcpyAsync(out, P.b.u, nvals * sizeof(double), cudaMemcpyDefault, s);
    }
  }

  static cudaError_t means(const void* pv, double* out, cudaStream_t s) {
    const KParams<real>& P = *static_cast<const KParams<real>*>(pv);
    if constexpr (MIXED) {
      return cudaMemcpyAsync(out, P.b.umean, (size_t)M * P.m.ne * sizeof(double), cudaMemcpyDefault, s);
    } else {
      const int nthr = M * P.m.ne;
      k_element_means<DIM, N, M><<<(nthr + kRowsPerBlock - 1) / kRowsPerBlock, kRowsPerBlock, 0, s>>>(
          P.b.u, out, P.m.ne, P.td);
      return cudaGetLastError();
    }
  }

  static const KernelSet* set() {
    static const KernelSet ks = {DIM, N, M, NP, MIXED ? 1 : 0, 4, &step,
                                 {&launch_local, &launch_face, &launch_update, &launch_finish},
                                 {"k_local", "k_face", "k_update", "k_finish_step"},
                                 &prologue, &split, &join, &means, &configure};
    return &ks;
  }
};

// Registries, one per translation unit (equation x dimension).
const KernelSet* kernels_linadv1d(int N, int mixed);
const KernelSet* kernels_linadv2d(int N, int mixed);
const KernelSet* kernels_euler1d(int N, int mixed);
const KernelSet* kernels_euler2d(int N, int mixed);
const KernelSet* kernels_tenmoment1d(int N, int mixed);
const KernelSet* kernels_tenmoment2d(int N, int mixed);
const KernelSet* kernels_burgers1d(int N, int mixed);
const KernelSet* kernels_varadv1d(int N, int mixed);
const KernelSet* kernels_euler1d_grav(int N, int mixed);
const KernelSet* kernels_euler2d_grav(int N, int mixed);

}  // namespace crk
