// fix_y.cu -- the FP64 complex FFT along y in block fixed point
// (chanfs_fix.cuh), and the cosine / sine transforms of walls in y on top of it.
//
// A CTA takes tk neighbouring complex columns of one z plane (rows of 16 tk
// contiguous bytes; consecutive threads on consecutive columns), every column
// with its own scale.  The first pass reads its butterflies from global memory
// into registers, the last one writes them back, so a tile visits shared
// memory only between passes.  512 x 384 x 384 on GB300: 1.70 ms in FP64 on TMA
// tiles (bound by the FP64 pipe), 0.43 ms here (2.8 TB/s), bound by the integer
// ALU pipe and by the barriers between the passes of a tile; 3456 x 3072 x 30 11 ms
// and 3.7 ms (tiles of two columns, one CTA of 24 warps per SM).
#include "chanfs_fix.cuh"
#include "chanfs_internal.cuh"

namespace chanfs {

struct YTile {
  double2* col;    // column 0 of the tile, row 0 of the plane
  int M;           // columns of the field (row stride)
  int valid;       // columns of this tile inside it
  int tk, sh;      // columns of the tile (a power of two), its logarithm
  int n, headroom, growth, div;
  int drop;        // 2^-drop: the passes' divisions
  bool first;      // the tile holds the packed column kx = 0
  Fix *A, *B;
  unsigned *top, *most, *quanta;
  FixScale* scale;
};

// Rows of a wall transform: element t of the FFT is row wall_row(t).
__device__ __forceinline__ int wall_row(int t, int n) {
  return t < (n + 1) / 2 ? 2 * t : 2 * (n - 1 - t) + 1;
}

enum { kPeriodic = 0, kCos = 1, kSin = 2 };

// Element e of column c of the first pass's input.
template <bool INV, bool WALL>
__device__ __forceinline__ double2 load_elem(const YTile& t, int e, int c, int ytype) {
  const double2* p = t.col + c;
  if constexpr (WALL && !INV) {
    const int j = wall_row(e, t.n);
    double2 v = p[(size_t)j * t.M];
    if (ytype == kSin && (j & 1)) v = make_double2(-v.x, -v.y);
    return v;
  } else if constexpr (WALL) {
    return p[(size_t)(ytype == kSin ? t.n - 1 - e : e) * t.M];  // X_e
  } else {
    return p[(size_t)e * t.M];
  }
}

// The packed column kx = 0 is stored untangled (slot ky holds F(0, ky), slot Ny -
// ky holds F(Nx/2, ky)): Z_ky = F0 + i FM, Z_{Ny-ky} = conj F0 + i conj FM.
__device__ __forceinline__ double2 load_packed(const YTile& t, int e) {
  const int n = t.n;
  const double2 v = t.col[(size_t)e * t.M];
  if (e == 0 || 2 * e == n) return v;
  const double2 w = t.col[(size_t)(n - e) * t.M];
  return 2 * e < n ? make_double2(v.x - w.y, v.y + w.x) : make_double2(w.x + v.y, v.x - w.y);
}

// Point e of column c as the first pass reads it.
template <bool INV, bool WALL>
__device__ __forceinline__ double2 load_point(const YTile& t, int e, int c, int ytype) {
  if (INV && !WALL && t.first && c == 0) return load_packed(t, e);
  return load_elem<INV, WALL>(t, e, c, ytype);
}

// V_e of the inverse wall transform from its column's X: conj(w_e) (X_e - i
// X_{N-e}), w_e = exp(-i pi e / 2N); V_0 = X_0.  (Points past the middle: w_m
// (X_e + ... ) with m = N - e, the same formula.)
__device__ __forceinline__ Fix wall_unmix(Fix xe, Fix xn, int4 wconj) {
  return fmul(Fix{xe.x + xn.y, xe.y - xn.x}, wconj);
}

// The first pass of a tile: at most one item per thread, kept in registers from
// the scan of its magnitudes on.
template <int R> struct YItem {  // this thread's
  int c, j;
  bool on;
  __device__ __forceinline__ explicit YItem(const YTile& t) {
    const int it = threadIdx.x;
    c = it & (t.tk - 1);
    j = it >> t.sh;
    on = it < (t.n / R) << t.sh && c < t.valid;
  }
  template <bool INV, bool WALL>
  __device__ __forceinline__ double2 value(const YTile& t, int ytype, int r) const {
    return load_point<INV, WALL>(t, j + r * (t.n / R), c, ytype);
  }
  __device__ __forceinline__ int place(const YTile& t, int r) const {  // of result r, in A
    return fix_pad(((j * R + r) << t.sh) + c);
  }
};
// The columns' maxima from their threads' (to t.top and t.most); whether one of
// them may have to be moved (fix_move), the same to the whole tile.
__device__ __forceinline__ bool column_max(const YTile& t, int c, bool on, unsigned top, float sum) {
  const bool odd = on && !fix_near(top);
  unsigned most = __float_as_uint(sum);
  for (int o = t.tk; o < 32; o *= 2) {
    top = max(top, __shfl_xor_sync(~0u, top, o));
    most = max(most, __shfl_xor_sync(~0u, most, o));
  }
  if ((threadIdx.x & 31) < t.tk) {
    atomicMax(t.top + c, top);
    atomicMax(t.most + c, most);
  }
  return __syncthreads_or(odd);
}
// The scale of a thread's column, its values times 2^k (to t.scale for the others).
// (sums: whether it uses the sum over the column.)
template <int R>
__device__ __forceinline__ int first_scale(const YTile& t, const YItem<R>& it, float sum, int k,
                                           bool sums) {
  const int c = it.c;
  if (sums) {
    unsigned q = it.on ? fix_quanta(sum, t.top[c], t.most[c]) : 0u;
    for (int o = t.tk; o < 32; o *= 2) q += __shfl_xor_sync(~0u, q, o);
    if ((threadIdx.x & 31) < t.tk) atomicAdd(t.quanta + c, q);
    __syncthreads();
  }
  const FixScale f = fix_scale_of(t.top[c], t.most[c], t.quanta[c], t.growth, t.headroom, t.div);
  if (it.on && it.j == 0) t.scale[c] = fix_moved_back(f, k);
  return f.s;
}
// Point r of an item in fixed point, from its value x (times 2^k; the mirrored point
// of a wall is read here).
template <int R, bool INV, bool WALL>
__device__ __forceinline__ Fix first_point(const YTile& t, const YItem<R>& it, int ytype, int r,
                                           double2 x, int k, int s, const int4* __restrict__ wy) {
  const Fix v = fix_from(x, s);
  if constexpr (INV && WALL) {
    const int e = it.j + r * (t.n / R);
    if (e > 0) {
      double2 xn = load_elem<INV, WALL>(t, t.n - e, it.c, ytype);
      xn = fix_moved(xn, k);
      return wall_unmix(v, fix_from(xn, s), __ldg(wy + e));
    }
  }
  return v;
}
// The pass up to its points in fixed point, left at the item's places of A, for a
// tile with a column far from 1.  (A call that reads its values twice and keeps few
// registers: the schedule of the other tiles knows nothing of it.)
template <int R, bool INV, bool WALL>
static __device__ __noinline__ void first_far(YTile t, int ytype, bool sums,
                                              const int4* __restrict__ wy) {
  const YItem<R> it(t);
  const int k = fix_move(t.top[it.c]);  // from the first attempt
  __syncthreads();
  if (threadIdx.x < t.tk) t.top[it.c] = t.most[it.c] = 0u;
  __syncthreads();
  unsigned top = 0u;
  float sum = 0.0f;
  if (it.on)
#pragma unroll 1
    for (int r = 0; r < R; ++r)
      fix_gather(fix_moved(it.template value<INV, WALL>(t, ytype, r), k), top, sum);
  column_max(t, it.c, it.on, top, sum);
  const int s = first_scale<R>(t, it, sum, k, sums);
  if (it.on)
#pragma unroll 1
    for (int r = 0; r < R; ++r) {
      const double2 x = fix_moved(it.template value<INV, WALL>(t, ytype, r), k);
      t.A[it.place(t, r)] = first_point<R, INV, WALL>(t, it, ytype, r, x, k, s, wy);
    }
}
template <int R, bool INV, bool WALL>
__device__ __forceinline__ void first_pass(const YTile& t, int ytype, bool sums,
                                           const int4* __restrict__ wy) {
  const YItem<R> it(t);
  double2 raw[R];
  unsigned top = 0u;
  float sum = 0.0f;
  if (it.on) {
    if (INV && !WALL && t.first && it.c == 0) {
      for (int r = 0; r < R; ++r) raw[r] = load_packed(t, it.j + r * (t.n / R));
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r)
        raw[r] = load_elem<INV, WALL>(t, it.j + r * (t.n / R), it.c, ytype);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) fix_gather(raw[r], top, sum);
  }
  __syncthreads();  // the reduction's cells are cleared
  Fix v[R];
  if (column_max(t, it.c, it.on, top, sum) &&
      __syncthreads_or(it.on && fix_far<R>(t.top[it.c], raw))) {
    first_far<R, INV, WALL>(t, ytype, sums, wy);
    if (!it.on) return;
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = t.A[it.place(t, r)];
  } else {
    const int s = first_scale<R>(t, it, sum, 0, sums);
    if (!it.on) return;
#pragma unroll
    for (int r = 0; r < R; ++r)
      v[r] = first_point<R, INV, WALL>(t, it, ytype, r, raw[r], 0, s, wy);
  }
  fdft<R, INV>(v);
#pragma unroll
  for (int r = 0; r < R; ++r) t.A[it.place(t, r)] = v[r];
}

template <int R, bool INV, bool HALF>
__device__ __forceinline__ void middle_pass(const YTile& t, const Fix* in, Fix* out, int L,
                                            const int4* __restrict__ tw) {
  const int Q = t.n / R, items = Q << t.sh;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int c = it & (t.tk - 1), j = it >> t.sh;
    const int sh = t.sh;
    fix_butterfly<R, INV, HALF>(in, out, j, Q, L, tw, [=](int e) { return fix_pad((e << sh) + c); });
  }
}

// The last pass: plain columns to global memory.  A forward wall transform
// leaves every column in shared memory for the mixing pass, the tile of the
// packed column leaves that one.
template <int R, bool INV, bool WALL, bool HALF>
__device__ __forceinline__ void last_pass(const YTile& t, const Fix* in, Fix* keep, int ytype,
                                          const int4* __restrict__ tw) {
  const int n = t.n, Q = n / R, items = Q << t.sh;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int c = it & (t.tk - 1), j = it >> t.sh;
    if (c >= t.valid) continue;
    Fix v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = in[fix_pad(((j + r * Q) << t.sh) + c)];
    fix_twiddle_dft<R, INV, HALF>(v, tw + j, Q);
    if (!INV && (WALL || (t.first && c == 0))) {
#pragma unroll
      for (int r = 0; r < R; ++r) keep[fix_pad(((j + r * Q) << t.sh) + c)] = v[r];
    } else {
      const FixScale f = t.scale[c];
      double2* o = t.col + c;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int e = j + r * Q;
        double2 z = fix_to(v[r], f.s - t.drop, f.kind);
        int row = e;
        if constexpr (WALL) {
          row = wall_row(e, n);
          if (ytype == kSin && (row & 1)) z = make_double2(-z.x, -z.y);
        }
        o[(size_t)row * t.M] = z;
      }
    }
  }
}

// The forward wall transform from V: with A = w_k V_k, B = conj(w_k) V_{N-k},
// 2 X_k = A + B and 2 X_{N-k} = i (A - B); X_0 = V_0.
__device__ __forceinline__ void wall_mix(const YTile& t, const Fix* in, int ytype,
                                         const int4* __restrict__ wy) {
  const int n = t.n, items = (n / 2 + 1) << t.sh;
  for (int it = threadIdx.x; it < items; it += blockDim.x) {
    const int c = it & (t.tk - 1), k = it >> t.sh;
    if (c >= t.valid) continue;
    const FixScale f = t.scale[c];
    double2* o = t.col + c;
    const auto slot = [&](int e) { return (size_t)(ytype == kSin ? n - 1 - e : e) * t.M; };
    const Fix vk = in[fix_pad((k << t.sh) + c)];
    if (k == 0) {
      o[slot(0)] = fix_to(vk, f.s - t.drop, f.kind);
      continue;
    }
    const int4 w = __ldg(wy + k);
    const Fix a = fmul(vk, w);
    const Fix b = fmul(in[fix_pad(((n - k) << t.sh) + c)], make_int4(w.x, w.y, -w.z, -w.w));
    o[slot(k)] = fix_to(fadd(a, b), f.s - t.drop + 1, f.kind);
    if (n - k != k) o[slot(n - k)] = fix_to(Fix{b.y - a.y, a.x - b.x}, f.s - t.drop + 1, f.kind);
  }
}

// The packed column kx = 0 of the forward transform: slot ky (0 < 2 ky < Ny)
// takes F(0, ky) = (Z_ky + conj Z_{Ny-ky}) / 2, slot Ny - ky takes F(Nx/2, ky)
// = -i (Z_ky - conj Z_{Ny-ky}) / 2; the self-conjugate slots keep the pair.
__device__ __forceinline__ void untangle_column(const YTile& t, const Fix* in) {
  const int n = t.n;
  const FixScale f = t.scale[0];
  for (int k = threadIdx.x; 2 * k <= n; k += blockDim.x) {
    const Fix z = in[fix_pad(k << t.sh)];
    if (k == 0 || 2 * k == n) {
      t.col[(size_t)k * t.M] = fix_to(z, f.s - t.drop, f.kind);
      continue;
    }
    const Fix m = in[fix_pad((n - k) << t.sh)];
    t.col[(size_t)k * t.M] = fix_to(Fix{z.x + m.x, z.y - m.y}, f.s - t.drop + 1, f.kind);
    t.col[(size_t)(n - k) * t.M] = fix_to(Fix{z.y + m.y, m.x - z.x}, f.s - t.drop + 1, f.kind);
  }
}

template <int N, bool INV, int P>
__device__ __forceinline__ void fixed_middle(const YTile& t, Fix* a, Fix* b, const int4* tw,
                                             Fix** end) {
  if constexpr (P + 1 < fix_npass<false>(N)) {
    middle_pass<fix_rad<false, INV>(N, P), INV, false>(t, a, b, fix_span<false, INV>(N, P),
                                                tw + fix_twoff<false, INV>(N, P));
    __syncthreads();
    fixed_middle<N, INV, P + 1>(t, b, a, tw, end);
  } else {
    *end = a;
  }
}

// Columns per tile (a power of two, as its logarithm): 8, rows of 128 bytes,
// while the first pass's items (`items` per column) fit 384 threads, else 4, and
// fewer only past 768 threads (rows of 32 and 16 bytes cost more than the waiting
// of one large CTA per SM).
__host__ __device__ constexpr int y_shift(int items) {
  int sh = 3;
  while (sh > 0 && (items << sh) > (sh == 3 ? 384 : 768)) --sh;
  return sh;
}
constexpr int y_threads(int n) {
  const int items = n / fix_radix<false>(n, 0);
  return ((items << y_shift(items)) + 31) / 32 * 32;
}

constexpr size_t y_smem(int n, int sh) {
  const size_t pts = (size_t)n << sh;
  return 2 * (pts + (pts >> 3)) * sizeof(Fix) + ((size_t)5 << sh) * sizeof(unsigned);
}
// Launch bounds: 24 warps per SM (80 registers), or 28 (72) where that and shared
// memory make room for a block more (108, 144, 216 and lengths up to 72: 216 forward
// 37 us with three blocks of nine warps, 41 with two).
constexpr bool y_tight(int n) {
  const int warps = y_threads(n) / 32;
  const int room = (int)(228 * 1024 / (y_smem(n, y_shift(n / fix_radix<false>(n, 0))) + 1024));
  return room > 24 / warps && 28 / warps > 24 / warps;
}
// N > 0: the compile-time length (periodic y); N = 0: any length, from d; N =
// kHalved: one whose radix-3 passes divide by 2.
template <int N, bool INV, bool WALL>
__global__ void __launch_bounds__(N <= 0 ? 768 : y_tight(N > 0 ? N : 9) ? 448 : y_threads(N > 0 ? N : 9),
                                  N <= 0                      ? 1
                                  : y_tight(N > 0 ? N : 9) ? 2
                                                              : 768 / y_threads(N > 0 ? N : 9))
    fix_y_kernel(double2* data, int M, FixDesc d, const int4* __restrict__ tw,
                 const int4* __restrict__ wy, int shift, int ytype) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr bool HALF = N == kHalved;
  const int n = N > 0 ? N : d.n;
  const int npass = N > 0 ? fix_npass<false>(N > 0 ? N : 8) : d.npass;
  const int sh =
      N > 0 ? y_shift((N > 0 ? N : 9) / fix_radix<false>(N > 0 ? N : 9, 0)) : shift;
  YTile t;
  t.n = n;
  t.M = M;
  t.sh = sh;
  t.tk = 1 << sh;
  const int x0 = blockIdx.x << sh;
  t.valid = min(t.tk, M - x0);
  t.first = x0 == 0;
  t.col = data + (size_t)blockIdx.y * n * M + x0;
  // (an inverse wall transform's V_e is up to |X_e| + |X_{N-e}|)
  t.headroom = INV && WALL ? 60 : 61;
  t.growth = N > 0 ? fix_growth<false, INV>(N > 0 ? N : 9) : d.growth;
  t.div = HALF ? d.div : 2;
  t.drop = HALF ? d.drop : 2 * (npass - 1);
  const int pts = n << sh, buf = pts + (pts >> 3);
  t.A = reinterpret_cast<Fix*>(smem_raw);
  t.B = t.A + buf;
  t.top = reinterpret_cast<unsigned*>(t.B + buf);
  t.most = t.top + t.tk;
  t.quanta = t.most + t.tk;
  t.scale = reinterpret_cast<FixScale*>(t.quanta + t.tk);
  for (int e = threadIdx.x; e < 3 * t.tk; e += blockDim.x) t.top[e] = 0u;
  Fix *a = t.A, *b = t.B;
  if constexpr (N > 0) {
    first_pass<fix_rad<false, INV>(N, 0), INV, false>(t, ytype, fix_uses_sum<false, INV>(N),
                                                             wy);
    __syncthreads();
    fixed_middle<N, INV, 1>(t, t.A, t.B, tw, &a);
    b = a == t.A ? t.B : t.A;
    constexpr int PL = fix_npass<false>(N) - 1;
    last_pass<fix_rad<false, INV>(N, PL), INV, false, false>(t, a, b, ytype,
                                                             tw + fix_twoff<false, INV>(N, PL));
  } else {
    switch (d.radix[0]) {
      case 8:
        if constexpr (!HALF) first_pass<8, INV, WALL>(t, ytype, d.sums, wy);
        break;
      case 6: first_pass<6, INV, WALL>(t, ytype, d.sums, wy); break;
      case 4:
        if constexpr (!HALF) first_pass<4, INV, WALL>(t, ytype, d.sums, wy);
        break;
      case 3: first_pass<3, INV, WALL>(t, ytype, d.sums, wy); break;
      default:
        if constexpr (!HALF) first_pass<2, INV, WALL>(t, ytype, d.sums, wy);
        break;
    }
    __syncthreads();
    for (int p = 1; p + 1 < npass; ++p) {
      const int L = d.span[p];
      const int4* w = tw + d.twoff[p];
      switch (d.radix[p]) {
        case 8:
          if constexpr (!HALF) middle_pass<8, INV, false>(t, a, b, L, w);
          break;
        case 6: middle_pass<6, INV, false>(t, a, b, L, w); break;
        case 4:
          if constexpr (!HALF) middle_pass<4, INV, false>(t, a, b, L, w);
          break;
        case 3: middle_pass<3, INV, HALF>(t, a, b, L, w); break;
        default:
          if constexpr (!HALF) middle_pass<2, INV, false>(t, a, b, L, w);
          break;
      }
      __syncthreads();
      Fix* s = a;
      a = b;
      b = s;
    }
    const int4* w = tw + d.twoff[npass - 1];
    switch (d.radix[npass - 1]) {
      case 8:
        if constexpr (!HALF) last_pass<8, INV, WALL, false>(t, a, b, ytype, w);
        break;
      case 6: last_pass<6, INV, WALL, false>(t, a, b, ytype, w); break;
      case 4:
        if constexpr (!HALF) last_pass<4, INV, WALL, false>(t, a, b, ytype, w);
        break;
      case 3: last_pass<3, INV, WALL, HALF>(t, a, b, ytype, w); break;
      default:
        if constexpr (!HALF) last_pass<2, INV, WALL, false>(t, a, b, ytype, w);
        break;
    }
  }
  if constexpr (!INV) {
    if (WALL || t.first) {
      __syncthreads();
      if constexpr (WALL) wall_mix(t, b, ytype, wy);
      else untangle_column(t, b);
    }
  }
}

template <int N, bool INV, bool WALL>
static cudaError_t go(const cfs_plan* P, double* data, int sh, int threads, cudaStream_t st) {
  auto k = fix_y_kernel<N, INV, WALL>;
  allow_max_smem(k);
  const dim3 grid((P->M + (1 << sh) - 1) >> sh, P->nz);
  k<<<grid, threads, y_smem(P->ny, sh), st>>>(
      reinterpret_cast<double2*>(data), P->M, INV ? P->yinv : P->yfwd, INV ? P->d_yinv : P->d_yfwd,
      INV ? P->d_ywall_inv : P->d_ywall, sh, P->ybc);
  return cudaGetLastError();
}

template <bool INV, bool WALL>
static cudaError_t dispatch(const cfs_plan* P, double* data, cudaStream_t st) {
  const int n = P->ny;
  const int T = n / (INV ? P->yinv : P->yfwd).radix[0];  // items per column, at most 729
  const int sh = y_shift(T);
  const int threads = ((T << sh) + 31) / 32 * 32;
  if constexpr (!WALL) {
    switch (n) {
#define CHANFS_FIX_LEN(n) \
  case n:                 \
    return go<n, INV, false>(P, data, sh, threads, st);
      CHANFS_FIX_LENGTHS
      CHANFS_FIX_LEN(2304) CHANFS_FIX_LEN(3072) CHANFS_FIX_LEN(3456) CHANFS_FIX_LEN(4096)
#undef CHANFS_FIX_LEN
      default: break;
    }
  }
  if (P->yfwd.half) return go<kHalved, INV, WALL>(P, data, sh, threads, st);
  return go<0, INV, WALL>(P, data, sh, threads, st);
}

cudaError_t launch_fix_y(const cfs_plan* P, double* data, bool inverse, cudaStream_t st) {
  if (P->ybc == CFS_Y_PERIODIC)
    return inverse ? dispatch<true, false>(P, data, st) : dispatch<false, false>(P, data, st);
  return inverse ? dispatch<true, true>(P, data, st) : dispatch<false, true>(P, data, st);
}

}  // namespace chanfs
