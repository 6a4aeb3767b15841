// helm_thomas.cu -- the z-implicit Helmholtz systems (I - c L_z) u = rhs of
// Eq. 11 by a plain Thomas sweep per (x, y) column, the alternative to the
// paper's Algorithm 2 that the tuner may pick per size.
//
// Every column has the same coefficients, so the LU factors are computed
// once per (c, loc) on the host (beside Algorithm 2's Step 1):
//   fs_k = 1/piv_k, fa_k = A'_k/piv_k, fc_k = C'_k/piv_k,
//   piv_0 = B'_0, piv_k = B'_k - A'_k fc_{k-1},
// and a sweep is g_k = fs_k d_k - fa_k g_{k-1} up the column (g written to
// u), then u_k = g_k - fc_k u_{k+1} back down: 3 instructions per unknown
// against Algorithm 2's 5, for twice the field traffic (g goes through
// memory).  One thread per column, consecutive threads on consecutive x, so
// every z-row access of a warp is one contiguous run; each thread loads the
// next group of rows of its column while it sweeps one (the sweep is sequential in
// z), and the factors sit in shared memory.  rhs == u is allowed: the forward sweep
// reads a row before it writes it.
// Bound by the FP64 pipe (3 instructions per unknown at 528 G/s, 430 us at 512 x 384
// x 384: 481 us here).  Two neighbouring columns per thread measured slower (509 us
// there, 129 against 107 at 512 x 162 x 192, groups of boxes 4 to 14 %), as did
// groups of four rows (107 and 110 at the latter).
#include "chanfs_group.cuh"

namespace chanfs {

constexpr int kHThBlock = 128;  // columns per block

// Rows per group (two groups are in flight).
template <class R> struct hth_rows { static constexpr int value = 8; };
template <> struct hth_rows<float> { static constexpr int value = 12; };

template <class R>
__device__ __forceinline__ void helm_thomas_body(const R* rhs, R* u, const R* __restrict__ fac,
                                                 long long ncols, int n, int nz, int face,
                                                 long long blk) {
  extern __shared__ __align__(16) unsigned char hth_smem[];
  R* sf = reinterpret_cast<R*>(hth_smem);  // fs | fa | fc
  for (int i = threadIdx.x; i < 3 * n; i += blockDim.x) sf[i] = fac[i];
  __syncthreads();
  const long long col = blk * blockDim.x + threadIdx.x;
  if (col >= ncols) return;
  constexpr int G = hth_rows<R>::value;
  const R* fs = sf;
  const R* fa = sf + n;
  const R* fc = sf + 2 * n;
  R A[G], B[G];
  // f(i) for the rows k + i < n of a group.  (The break makes branches: rows past the
  // end, merely predicated off, took their time on the FP64 pipe all the same: 133
  // against 107 us for nine rows of 2048 x 1024 columns.)
  const auto by_group = [n](int k, auto f) {
    if (k + G <= n) {
#pragma unroll
      for (int i = 0; i < G; ++i) f(i);
    } else {
#pragma unroll
      for (int i = 0; i < G; ++i) {
        if (k + i >= n) break;
        f(i);
      }
    }
  };

  {  // forward: g_k = fs_k d_k - fa_k g_{k-1}
    const R* p = rhs + col;
    R* w = u + col;
    R g = R(0);
    const auto load = [&](R* q, int k) {
      by_group(k, [&](int i) {
        q[i] = *p;
        p += ncols;
      });
    };
    const auto run = [&](const R* q, int k) {
      by_group(k, [&](int i) {
        g = fma(-fa[k + i], g, fs[k + i] * q[i]);
        *w = g;
        w += ncols;
      });
    };
    load(A, 0);
    for (int k = 0; k < n; k += 2 * G) {
      load(B, k + G);
      run(A, k);
      load(A, k + 2 * G);
      run(B, k + G);
    }
  }
  {  // backward: u_{n-1} = g_{n-1}, u_k = g_k - fc_k u_{k+1}; r rows from the top
    const R* p = u + (long long)(n - 1) * ncols + col;
    R* w = u + (long long)(n - 1) * ncols + col;
    R x = R(0);
    const auto load = [&](R* q, int r) {
      by_group(r, [&](int i) {
        q[i] = *p;
        p -= ncols;
      });
    };
    const auto run = [&](const R* q, int r) {
      by_group(r, [&](int i) {
        x = fma(-fc[n - 1 - r - i], x, q[i]);
        *w = x;
        w -= ncols;
      });
    };
    load(A, 0);
    for (int r = 0; r < n; r += 2 * G) {
      load(B, r + G);
      run(A, r);
      load(A, r + 2 * G);
      run(B, r + G);
    }
  }
  if (face) u[(long long)(nz - 1) * ncols + col] = R(0);  // the wall slot
}

template <class R>
__global__ void __launch_bounds__(kHThBlock) helm_thomas_kernel(const R* rhs, R* u,
                                                                const R* __restrict__ fac,
                                                                long long ncols, int n, int nz,
                                                                int face) {
  helm_thomas_body<R>(rhs, u, fac, ncols, n, nz, face, blockIdx.x);
}

template <class R>
__global__ void __launch_bounds__(kHThBlock) helm_thomas_group_kernel(const HThomasBox* boxes,
                                                                      GroupMap g,
                                                                      const GroupIo* io) {
  int b, blk;
  if (!group_block(g, &b, &blk)) return;
  const HThomasBox& x = boxes[b];
  // per-call fields (FP64 boxes) come from the call's table; FP32 inner
  // solves work in place on the plan's residual field
  const R* rhs = x.per_call ? reinterpret_cast<const R*>(io[b].f) : static_cast<const R*>(x.rhs);
  R* u = x.per_call ? reinterpret_cast<R*>(io[b].p) : static_cast<R*>(x.u);
  helm_thomas_body<R>(rhs, u, static_cast<const R*>(x.fac), x.ncols, x.n, x.nz, x.face, blk);
}

template <class R>
static cudaError_t launch_t(const cfs_plan* P, const HelmCoef& h, const R* fac, const R* rhs,
                            R* u, cudaStream_t st) {
  const long long ncols = (long long)P->nx * P->ny;
  const unsigned grid = (unsigned)((ncols + kHThBlock - 1) / kHThBlock);
  const size_t smem = 3 * sizeof(R) * (size_t)h.n;
  auto k = helm_thomas_kernel<R>;
  allow_max_smem(k);
  k<<<grid, kHThBlock, smem, st>>>(rhs, u, fac, ncols, h.n, P->nz, h.loc == CFS_LOC_FACE);
  return cudaGetLastError();
}

cudaError_t launch_helm_thomas(const cfs_plan* P, const HelmCoef& h, const double* rhs,
                               double* u, cudaStream_t st) {
  return launch_t<double>(P, h, h.d_th, rhs, u, st);
}

cudaError_t launch_helm_thomas32(const cfs_plan* P, const HelmCoef& h, const float* rhs,
                                 float* u, cudaStream_t st) {
  if (!h.d_th32) return cudaErrorInvalidValue;  // FP64 plans hold no FP32 factors
  return launch_t<float>(P, h, h.d_th32, rhs, u, st);
}

size_t helm_thomas_group_box(const cfs_plan* P, const HelmCoef& h, bool fp32, HThomasBox* box,
                             int* blocks) {
  box->ncols = (long long)P->nx * P->ny;
  box->n = h.n;
  box->nz = P->nz;
  box->face = h.loc == CFS_LOC_FACE;
  box->per_call = !fp32;
  box->rhs = fp32 ? static_cast<const void*>(P->d_r32) : nullptr;
  box->u = fp32 ? static_cast<void*>(P->d_r32) : nullptr;
  box->fac = fp32 ? static_cast<const void*>(h.d_th32) : static_cast<const void*>(h.d_th);
  *blocks = (int)((box->ncols + kHThBlock - 1) / kHThBlock);
  return 3 * (fp32 ? sizeof(float) : sizeof(double)) * (size_t)h.n;
}

cudaError_t launch_helm_thomas_group(const HThomasBox* boxes, GroupMap g, int total, size_t smem,
                                     bool fp32, const GroupIo* io, cudaStream_t st) {
  if (total <= 0) return cudaSuccess;
  if (fp32) {
    auto k = helm_thomas_group_kernel<float>;
    allow_max_smem(k);
    k<<<total, kHThBlock, smem, st>>>(boxes, g, io);
  } else {
    auto k = helm_thomas_group_kernel<double>;
    allow_max_smem(k);
    k<<<total, kHThBlock, smem, st>>>(boxes, g, io);
  }
  return cudaGetLastError();
}

}  // namespace chanfs
