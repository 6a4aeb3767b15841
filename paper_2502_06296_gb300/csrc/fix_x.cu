// fix_x.cu -- the FP64 real FFT along x in block fixed point (chanfs_fix.cuh),
// packed output (App. A of the paper).
//
// A line of nx = 2M reals is M complex numbers; a thread takes one butterfly
// of the first pass straight from global memory into registers and one pair of
// mirrored butterflies of the last pass straight back, so that the line visits
// shared memory only between passes.  The last forward pass (the first inverse
// one) holds the butterflies i and Q - i together: their outputs (inputs) k
// and M - k are the pairs that the real transform untangles,
//   2 X_k = E - i W^k O,  2 X_{M-k} = conj(E + i W^k O),
//   E = Z_k + conj Z_{M-k},  O = Z_k - conj Z_{M-k},  W = exp(-2 pi i / nx).
// Item i = 0 holds the butterflies 0 and Q/2, whose pairs lie within each.
// What bounds it: the integer ALU pipe (about 57 of its instructions per real
// point: 21 in additions, 17 in the conversion from double, the rest in the
// products' halves; 68 % busy in ncu at 24 warps per SM), against 13.75
// instructions per point on an FP64 pipe 32 times narrower: 2.03 / 1.99 ms forward
// / inverse in FP64 at 512 x 384 x 384 on GB300, 0.33 / 0.32 ms here (3.7 TB/s).
// Lengths with up to three factors 3 are compiled with every radix, span and offset a constant;
// with a power of two of items per line, at most 32, a warp owns its lines and
// never waits for another.
#include "chanfs_fix.cuh"
#include "chanfs_internal.cuh"

namespace chanfs {

// Pairs of item i: entry r is (p[r], q[r]) = (Z_k, Z_{M-k}), k = pair_index.
template <int R>
__device__ __forceinline__ void pair_take(bool zero, const Fix* a, const Fix* b, Fix* p, Fix* q) {
#pragma unroll
  for (int r = 0; r < R; ++r) {
    p[r] = a[r];
    q[r] = b[R - 1 - r];
  }
  if (zero) {
    if constexpr (R == 6) {
      p[0] = q[0] = a[3];
      q[1] = a[5];
      q[2] = a[4];
      p[3] = b[0];
      q[3] = b[5];
      p[4] = b[1];
      q[4] = b[4];
      p[5] = b[2];
      q[5] = b[3];
    } else if constexpr (R == 4) {
      p[0] = q[0] = a[2];
      q[1] = a[3];
      p[2] = b[0];
      q[2] = b[3];
      p[3] = b[1];
      q[3] = b[2];
    } else if constexpr (R == 3) {
      p[0] = q[0] = b[1];
      q[1] = a[2];
      p[2] = b[0];
      q[2] = b[2];
    } else {
      p[0] = q[0] = a[1];
      p[1] = b[0];
      q[1] = b[1];
    }
  }
}
// The inverse of pair_take (a[0] of item 0 is set by the caller).
template <int R>
__device__ __forceinline__ void pair_give(bool zero, const Fix* p, const Fix* q, Fix* a, Fix* b) {
#pragma unroll
  for (int r = 0; r < R; ++r) {
    a[r] = p[r];
    b[R - 1 - r] = q[r];
  }
  if (zero) {
    if constexpr (R == 6) {
      a[1] = p[1];
      a[2] = p[2];
      a[3] = p[0];
      a[4] = q[2];
      a[5] = q[1];
      b[0] = p[3];
      b[1] = p[4];
      b[2] = p[5];
      b[3] = q[5];
      b[4] = q[4];
      b[5] = q[3];
    } else if constexpr (R == 4) {
      a[1] = p[1];
      a[2] = p[0];
      a[3] = q[1];
      b[0] = p[2];
      b[1] = p[3];
      b[2] = q[3];
      b[3] = q[2];
    } else if constexpr (R == 3) {
      a[1] = p[1];
      a[2] = q[1];
      b[0] = p[2];
      b[1] = p[0];
      b[2] = q[2];
    } else {
      a[1] = p[0];
      b[0] = p[1];
      b[1] = q[1];
    }
  }
}
template <int R> __device__ __forceinline__ int pair_index(bool zero, int i, int r, int Q) {
  if (!zero) return i + r * Q;
  if constexpr (R == 6) return r == 0 ? 3 * Q : r <= 2 ? r * Q : Q / 2 + (r - 3) * Q;
  if constexpr (R == 4) return r == 0 ? 2 * Q : r == 1 ? Q : r == 2 ? Q / 2 : Q / 2 + Q;
  if constexpr (R == 3) return r == 0 ? Q + Q / 2 : r == 1 ? Q : Q / 2;
  return r == 0 ? Q : Q / 2;
}
// Whether entry r of item 0 belongs to the butterfly Q/2 (absent if Q is odd).
template <int R> __device__ __forceinline__ bool pair_second(int r) {
  return R == 6 ? r >= 3 : R == 4 ? r >= 2 : R == 3 ? r != 1 : r == 1;
}

// What a group of G threads (a warp, or the CTA) works on.
struct XGroup {
  int lane, G;         // this thread among them
  int nl;              // its lines
  long long line0;     // the first one
  long long nlines;    // lines of the field
  int n, ps, headroom, growth, div;
  int drop;            // 2^-drop: the passes' divisions (and the factor 2 of 2 X or 2 Z)
  Fix *A, *B;          // two buffers of nl padded lines
  unsigned *top, *most, *quanta;
  FixScale* scale;
};

template <bool WARP> __device__ __forceinline__ void group_sync() {
  if constexpr (WARP) __syncwarp();
  else __syncthreads();
}

template <bool WARP> __device__ __forceinline__ bool group_any(bool v) {
  if constexpr (WARP) return __any_sync(~0u, v);
  else return __syncthreads_or(v);
}

// The maxima over the T items of each line (item lane of the group in line lane
// / T) of the values' magnitudes and of the butterflies' sums, and the sum of
// their quanta: the same on every thread of a line.  line_max also says whether a
// line of the group may have to be moved (fix_move), the same to the whole group.
template <bool WARP, int T>
__device__ __forceinline__ bool warp_lead(const XGroup& g) {  // a warp's items share a line
  return T ? T % 32 == 0 : g.nl == 1;
}
template <bool WARP, int T>
__device__ __forceinline__ bool line_max(const XGroup& g, int l, bool on, unsigned& top,
                                         unsigned& most) {
  if constexpr (WARP && T == 32) {
    top = __reduce_max_sync(~0u, top);
    most = __reduce_max_sync(~0u, most);
    return !fix_near(top);
  } else if constexpr (WARP) {
#pragma unroll
    for (int o = 1; o < T; o *= 2) {
      top = max(top, __shfl_xor_sync(~0u, top, o));
      most = max(most, __shfl_xor_sync(~0u, most, o));
    }
    return __any_sync(~0u, !fix_near(top));
  } else {
    const bool odd = on && !fix_near(top);
    if (warp_lead<WARP, T>(g)) {
      top = __reduce_max_sync(~0u, top);
      most = __reduce_max_sync(~0u, most);
      on = on && (g.lane & 31) == 0;
    }
    if (on) {
      atomicMax(g.top + l, top);
      atomicMax(g.most + l, most);
    }
    const bool any = __syncthreads_or(odd);
    top = g.top[l];
    most = g.most[l];
    return any;
  }
}
template <bool WARP, int T>
__device__ __forceinline__ unsigned line_sum(const XGroup& g, int l, bool on, unsigned v) {
  if constexpr (WARP && T == 32) {
    return __reduce_add_sync(~0u, v);
  } else if constexpr (WARP) {
#pragma unroll
    for (int o = 1; o < T; o *= 2) v += __shfl_xor_sync(~0u, v, o);
    return v;
  } else {
    if (warp_lead<WARP, T>(g)) {
      v = __reduce_add_sync(~0u, v);
      on = on && (g.lane & 31) == 0;
    }
    if (on) atomicAdd(g.quanta + l, v);
    __syncthreads();
    return g.quanta[l];
  }
}

// Value r of item i of the first pass: forward, butterfly i of the line (R points i +
// r Q); inverse, the pairs of item i (2 R points, and the point 0 of item 0).
template <int R, bool INV>
__device__ __forceinline__ double2 item_value(const double2* line, int n, int Q, int i, int r) {
  if constexpr (!INV) {
    return line[i + r * Q];
  } else {
    const bool z = i == 0;
    if (r == 2 * R) return z ? line[0] : make_double2(0.0, 0.0);
    const int k = pair_index<R>(z, i, r / 2, Q);
    const bool have = !z || (Q & 1) == 0 || !pair_second<R>(r / 2);
    return have ? line[r % 2 ? n - k : k] : make_double2(0.0, 0.0);
  }
}

// The first pass's arithmetic on an item of values raw(r), written to buffer A.
template <int R, bool INV, class Raw>
__device__ __forceinline__ void first_item(const XGroup& g, Fix* line, int n, int Q, int i,
                                           Raw raw, int s,
                                           const int4* __restrict__ post) {
  if constexpr (!INV) {
    Fix v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = fix_from(raw(r), s);
    fdft<R, false>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) line[fix_pad(i * R + r)] = v[r];
  } else {
    const bool z = i == 0;
    Fix a[R], b[R], p[R], q[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {  // 2 Z_k = E + i conj(W^k) T, T = X_k - conj X_{M-k}
      const Fix xk = fix_from(raw(2 * r), s), xm = fix_from(raw(2 * r + 1), s);
      const Fix e = {xk.x + xm.x, xk.y - xm.y};
      const Fix u = fmul(Fix{xk.x - xm.x, xk.y + xm.y},
                         __ldg(post + pair_index<R>(z, i, r, Q)));
      p[r] = {e.x - u.y, e.y + u.x};
      q[r] = {e.x + u.y, u.x - e.y};
    }
    pair_give<R>(z, p, q, a, b);
    if (z) {
      const Fix x0 = fix_from(raw(2 * R), s);  // (X_0, X_M)
      a[0] = {x0.x + x0.y, x0.x - x0.y};
    }
    fdft<R, true>(a);
    fdft<R, true>(b);
    const int jb = z ? Q / 2 : Q - i;
#pragma unroll
    for (int r = 0; r < R; ++r) line[fix_pad(i * R + r)] = a[r];
    if (!z || (Q & 1) == 0) {
#pragma unroll
      for (int r = 0; r < R; ++r) line[fix_pad(jb * R + r)] = b[r];
    }
  }
}

// The first pass of the group's lines: at most one item per thread, kept in
// registers from the scan of its magnitudes on.
template <int R, bool INV, int T> struct XItem {  // this thread's
  static constexpr int kRaw = INV ? 2 * R + 1 : R;
  int Q, l, i;
  bool on;
  const double2* line;
  __device__ __forceinline__ XItem(const XGroup& g, const double2* in) {
    Q = g.n / R;
    const int per = T ? T : (INV ? (Q + 1) / 2 : Q);
    l = min(g.lane / per, g.nl - 1);
    i = g.lane - l * per;
    on = g.lane < g.nl * per && l < g.nlines - g.line0;
    line = in + (g.line0 + l) * g.n;
  }
  __device__ __forceinline__ double2 value(const XGroup& g, int r) const {
    return item_value<R, INV>(line, g.n, Q, i, r);
  }
};
// Its scale and arithmetic, the line's values times 2^k.  (sums: whether the scale
// uses the sum over the line.  Inverse: the two butterflies of an item are each
// bounded by twice its sum, one factor 2 of which is in the headroom.)
template <int R, bool INV, bool WARP, int T, class Raw>
__device__ __forceinline__ void first_arith(const XGroup& g, const XItem<R, INV, T>& it, Raw raw,
                                            unsigned top, unsigned most, float sum, int k,
                                            bool sums, const int4* __restrict__ post) {
  unsigned quanta = 0u;
  if (sums)
    quanta = line_sum<WARP, T>(g, it.l, it.on,
                               it.on ? (INV ? 2u : 1u) * fix_quanta(sum, top, most) : 0u);
  if (it.on) {
    const FixScale f = fix_scale_of(top, most, quanta, g.growth, g.headroom, g.div);
    if (it.i == 0) g.scale[it.l] = fix_moved_back(f, k);
    first_item<R, INV>(g, g.A + it.l * g.ps, g.n, it.Q, it.i, raw, f.s, post);
  }
}
// The pass again from its loads on, for a group with a line far from 1.  (A call that
// reads its values twice rather than keep them: the registers and the schedule of
// the others know nothing of it.)
template <int R, bool INV, bool WARP, int T>
static __device__ __noinline__ void first_pass_far(XGroup g, const double2* in, bool sums,
                                                   const int4* __restrict__ post) {
  using Item = XItem<R, INV, T>;
  const Item it(g, in);
  unsigned top = 0u, most = 0u;
  float sum = 0.0f;
  if constexpr (WARP) {
    if (it.on)
#pragma unroll 1
      for (int r = 0; r < Item::kRaw; ++r) fix_gather(it.value(g, r), top, sum);
    line_max<WARP, T>(g, it.l, it.on, top, most);
  } else {
    top = g.top[it.l];  // the line's, from the first attempt
    __syncthreads();
    if (it.on && it.i == 0) g.top[it.l] = g.most[it.l] = 0u;
    __syncthreads();
  }
  const int k = fix_move(top);
  const auto raw = [&](int r) { return fix_moved(it.value(g, r), k); };
  top = 0u;
  sum = 0.0f;
  if (it.on)
#pragma unroll 1
    for (int r = 0; r < Item::kRaw; ++r) fix_gather(raw(r), top, sum);
  most = __float_as_uint(sum);
  line_max<WARP, T>(g, it.l, it.on, top, most);
  first_arith<R, INV, WARP, T>(g, it, raw, top, most, sum, k, sums, post);
}
template <int R, bool INV, bool WARP, int T>
__device__ __forceinline__ void first_pass(const XGroup& g, const double2* in, bool sums,
                                           const int4* __restrict__ post) {
  using Item = XItem<R, INV, T>;
  const Item it(g, in);
  double2 raw[Item::kRaw];
  unsigned top = 0u;
  float sum = 0.0f;
  if (it.on) {
#pragma unroll
    for (int r = 0; r < Item::kRaw; ++r) raw[r] = it.value(g, r);
#pragma unroll
    for (int r = 0; r < Item::kRaw; ++r) fix_gather(raw[r], top, sum);
  }
  if constexpr (!WARP) __syncthreads();  // the reduction's cells are cleared
  unsigned most = __float_as_uint(sum);
  if (line_max<WARP, T>(g, it.l, it.on, top, most) &&
      group_any<WARP>(it.on && fix_far<Item::kRaw>(top, raw)))
    first_pass_far<R, INV, WARP, T>(g, in, sums, post);
  else
    first_arith<R, INV, WARP, T>(g, it, [&](int r) { return raw[r]; }, top, most, sum, 0, sums,
                                 post);
}

// A middle pass over the group's lines, from one buffer to the other.
template <int R, bool INV, bool HALF>
__device__ __forceinline__ void middle_pass(const XGroup& g, const Fix* in, Fix* out, int L,
                                            const int4* __restrict__ tw) {
  const int Q = g.n / R, items = g.nl * Q;
  for (int it = g.lane; it < items; it += g.G) {
    const int l = it / Q, j = it - l * Q;
    fix_butterfly<R, INV, HALF>(in + l * g.ps, out + l * g.ps, j, Q, L, tw,
                          [](int e) { return fix_pad(e); });
  }
}

// The last forward pass with the untangling: pairs to global memory.
template <int R, bool HALF>
__device__ __forceinline__ void last_forward(const XGroup& g, const Fix* in, double2* out,
                                             const int4* __restrict__ tw,
                                             const int4* __restrict__ post) {
  const int n = g.n, Q = n / R, per = (Q + 1) / 2, items = g.nl * per;
  const bool odd = Q & 1;
  for (int it = g.lane; it < items; it += g.G) {
    const int l = it / per, i = it - l * per;
    if (g.line0 + l >= g.nlines) continue;
    const bool z = i == 0;
    const int jb = z ? Q / 2 : Q - i;
    const Fix* x = in + l * g.ps;
    Fix a[R], b[R], p[R], q[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      a[r] = x[fix_pad(i + r * Q)];
      b[r] = x[fix_pad(jb + r * Q)];
    }
    fix_twiddle_dft<R, false, HALF>(a, tw + i, Q);
    fix_twiddle_dft<R, false, HALF>(b, tw + jb, Q);
    const FixScale f = g.scale[l];
    const int sh = f.s - g.drop;
    double2* o = out + (g.line0 + l) * n;
    if (z) o[0] = fix_to(Fix{a[0].x + a[0].y, a[0].x - a[0].y}, sh - 1, f.kind);  // (X_0, X_M)
    pair_take<R>(z, a, b, p, q);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (z && odd && pair_second<R>(r)) continue;
      const int k = pair_index<R>(z, i, r, Q);
      const Fix e = {p[r].x + q[r].x, p[r].y - q[r].y};
      const Fix u = fmul(Fix{p[r].x - q[r].x, p[r].y + q[r].y}, __ldg(post + k));
      o[k] = fix_to(Fix{e.x + u.y, e.y - u.x}, sh, f.kind);
      if (n - k != k) o[n - k] = fix_to(Fix{e.x - u.y, -e.y - u.x}, sh, f.kind);
    }
  }
}

static __device__ __noinline__ double2 scaled_by(double2 z, double mul) {
  return make_double2(z.x * mul, z.y * mul);
}

// The last inverse pass: plain butterflies to global memory.
// (The factor `mul`, where a caller wants one, goes on last: its FP64 products
// are kept out of the plain code, where they would be most of the FP64 work.)
template <int R, bool HALF>
__device__ __forceinline__ void last_inverse(const XGroup& g, const Fix* in, double2* out,
                                             const int4* __restrict__ tw, double mul, int scaled) {
  const int n = g.n, Q = n / R, items = g.nl * Q;
  for (int it = g.lane; it < items; it += g.G) {
    const int l = it / Q, j = it - l * Q;
    if (g.line0 + l >= g.nlines) continue;
    const Fix* x = in + l * g.ps;
    Fix v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = x[fix_pad(j + r * Q)];
    fix_twiddle_dft<R, true, HALF>(v, tw + j, Q);
    const FixScale f = g.scale[l];
    const int sh = f.s - g.drop;
    double2* o = out + (g.line0 + l) * n;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      double2 z = fix_to(v[r], sh, f.kind);
      if (scaled) z = scaled_by(z, mul);
      o[j + r * Q] = z;
    }
  }
}

// Items per line of the first pass.
template <bool INV> __host__ __device__ constexpr int x_items(int n) {
  const int R = fix_rad<true, INV>(n, 0), Q = n / R;
  return INV ? (Q + 1) / 2 : Q;
}
__host__ __device__ constexpr bool warp_lines(int items) {
  return items <= 32 && (items & (items - 1)) == 0;
}

template <int N, bool INV, int P>
__device__ __forceinline__ void fixed_middle(const XGroup& g, Fix* a, Fix* b, const int4* tw,
                                             Fix** end) {
  constexpr int NP = fix_npass<true>(N);
  constexpr bool WARP = warp_lines(x_items<INV>(N));
  if constexpr (P + 1 < NP) {
    middle_pass<fix_rad<true, INV>(N, P), INV, false>(g, a, b, fix_span<true, INV>(N, P),
                                                      tw + fix_twoff<true, INV>(N, P));
    group_sync<WARP>();
    fixed_middle<N, INV, P + 1>(g, b, a, tw, end);
  } else {
    *end = a;
  }
}

// N > 0: the compile-time length; N = 0: any length, from d (at most 384 items
// of the first pass per line); N = kHalved: one whose radix-3 passes divide by 2.
template <int N, bool INV>
__global__ void __launch_bounds__(N > 0 ? 256 : 384, N > 0 ? 3 : 2)
    fix_x_kernel(const double2* in, double2* out, long long nlines, FixDesc d,
                 const int4* __restrict__ tw, const int4* __restrict__ post, int lb, double mul,
                 int scaled) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int T = N > 0 ? x_items<INV>(N > 0 ? N : 8) : 0;
  constexpr bool WARP = N > 0 && warp_lines(T);
  constexpr bool HALF = N == kHalved;
  const int n = N > 0 ? N : d.n;
  const int ps = n + (n >> 3);
  XGroup g;
  g.n = n;
  g.ps = ps;
  // forward: 2 X is up to 4 times a value of the last pass; inverse: a butterfly
  // of 2 Z is up to twice its item's sum, and nothing follows the last pass
  g.headroom = INV ? 61 : 60;
  g.growth = N > 0 ? fix_growth<true, INV>(N > 0 ? N : 9) : d.growth;
  g.div = HALF ? d.div : 2;
  g.nlines = nlines;
  const int grp = WARP ? (int)(threadIdx.x >> 5) : 0;
  g.nl = WARP ? 32 / (T ? T : 32) : lb;
  g.lane = WARP ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
  g.G = WARP ? 32 : (int)blockDim.x;
  g.line0 = (long long)blockIdx.x * lb + grp * g.nl;
  Fix* buf = reinterpret_cast<Fix*>(smem_raw);
  g.A = buf + grp * g.nl * ps;
  const int npass = N > 0 ? fix_npass<true>(N > 0 ? N : 8) : d.npass;
  g.drop = (HALF ? d.drop : 2 * (npass - 1)) - 1;
  g.B = g.A + (npass > 2 ? lb * ps : 0);
  int* cells = reinterpret_cast<int*>(buf + (npass > 2 ? 2 : 1) * lb * ps);
  g.scale = reinterpret_cast<FixScale*>(cells) + grp * g.nl;
  g.top = reinterpret_cast<unsigned*>(cells + 2 * lb);
  g.most = g.top + lb;
  g.quanta = g.most + lb;
  if constexpr (!WARP)
    for (int e = threadIdx.x; e < 3 * lb; e += blockDim.x) g.top[e] = 0u;
  if constexpr (N > 0) {
    first_pass<fix_rad<true, INV>(N, 0), INV, WARP, T>(g, in, fix_uses_sum<true, INV>(N),
                                                              post);
    group_sync<WARP>();
    Fix* end;
    fixed_middle<N, INV, 1>(g, g.A, g.B, tw, &end);
    constexpr int PL = fix_npass<true>(N) - 1;
    if constexpr (INV)
      last_inverse<fix_rad<true, true>(N, PL), false>(
          g, end, out, tw + fix_twoff<true, true>(N, PL), mul, scaled);
    else
      last_forward<fix_rad<true, false>(N, PL), false>(
          g, end, out, tw + fix_twoff<true, false>(N, PL), post);
  } else {
    switch (d.radix[0]) {
      case 8:
        if constexpr (!INV && !HALF) first_pass<8, INV, false, 0>(g, in, d.sums, post);
        break;
      case 6: first_pass<6, INV, false, 0>(g, in, d.sums, post); break;
      case 4:
        if constexpr (!HALF) first_pass<4, INV, false, 0>(g, in, d.sums, post);
        break;
      case 3: first_pass<3, INV, false, 0>(g, in, d.sums, post); break;
      default:
        if constexpr (!HALF) first_pass<2, INV, false, 0>(g, in, d.sums, post);
        break;
    }
    __syncthreads();
    Fix *a = g.A, *b = g.B;
    for (int p = 1; p + 1 < npass; ++p) {
      const int L = d.span[p];
      const int4* t = tw + d.twoff[p];
      switch (d.radix[p]) {
        case 8:
          if constexpr (!HALF) middle_pass<8, INV, false>(g, a, b, L, t);
          break;
        case 6: middle_pass<6, INV, false>(g, a, b, L, t); break;
        case 4:
          if constexpr (!HALF) middle_pass<4, INV, false>(g, a, b, L, t);
          break;
        case 3: middle_pass<3, INV, HALF>(g, a, b, L, t); break;
        default:
          if constexpr (!HALF) middle_pass<2, INV, false>(g, a, b, L, t);
          break;
      }
      __syncthreads();
      Fix* s = a;
      a = b;
      b = s;
    }
    const int4* t = tw + d.twoff[npass - 1];
    switch (d.radix[npass - 1]) {
      case 8:
        if constexpr (INV && !HALF) last_inverse<8, false>(g, a, out, t, mul, scaled);
        break;
      case 6:
        if constexpr (INV) last_inverse<6, false>(g, a, out, t, mul, scaled);
        else last_forward<6, false>(g, a, out, t, post);
        break;
      case 4:
        if constexpr (HALF) break;
        else if constexpr (INV) last_inverse<4, false>(g, a, out, t, mul, scaled);
        else last_forward<4, false>(g, a, out, t, post);
        break;
      case 3:
        if constexpr (INV) last_inverse<3, HALF>(g, a, out, t, mul, scaled);
        else last_forward<3, HALF>(g, a, out, t, post);
        break;
      default:
        if constexpr (HALF) break;
        else if constexpr (INV) last_inverse<2, false>(g, a, out, t, mul, scaled);
        else last_forward<2, false>(g, a, out, t, post);
        break;
    }
  }
}

template <int N, bool INV>
static cudaError_t go(const cfs_plan* P, const double* in, double* out, double mul, long long nl,
                      int threads, int lb, cudaStream_t st) {
  const FixDesc& d = INV ? P->xinv : P->xfwd;
  const int n = P->M;
  const size_t smem = (size_t)(d.npass > 2 ? 2 : 1) * lb * (n + (n >> 3)) * sizeof(Fix) +
                      (size_t)lb * 5 * sizeof(int);
  auto k = fix_x_kernel<N, INV>;
  allow_max_smem(k);
  k<<<(unsigned)((nl + lb - 1) / lb), threads, smem, st>>>(
      reinterpret_cast<const double2*>(in), reinterpret_cast<double2*>(out), nl, d,
      INV ? P->d_xinv : P->d_xfwd, INV ? P->d_xpost_inv : P->d_xpost, lb, mul, mul != 1.0);
  return cudaGetLastError();
}

template <int N, bool INV>
static cudaError_t go_fixed(const cfs_plan* P, const double* in, double* out, double mul,
                            long long nl, cudaStream_t st) {
  constexpr int T = x_items<INV>(N);
  if constexpr (warp_lines(T)) {
    return go<N, INV>(P, in, out, mul, nl, 128, 4 * (32 / T), st);
  } else {
    constexpr int lb = T >= 192 ? 1 : 192 / T;
    return go<N, INV>(P, in, out, mul, nl, (lb * T + 31) / 32 * 32, lb, st);
  }
}

template <bool INV>
static cudaError_t dispatch(const cfs_plan* P, const double* in, double* out, double mul,
                            long long nl, cudaStream_t st) {
  switch (P->M) {
#define CHANFS_FIX_LEN(n) \
  case n:                 \
    return go_fixed<n, INV>(P, in, out, mul, nl, st);
    CHANFS_FIX_LENGTHS
#undef CHANFS_FIX_LEN
    default: break;
  }
  const int T = x_items<INV>(P->M), lb = T >= 192 ? 1 : 192 / T;
  const int threads = (lb * T + 31) / 32 * 32;
  if (P->xfwd.half) return go<kHalved, INV>(P, in, out, mul, nl, threads, lb, st);
  return go<0, INV>(P, in, out, mul, nl, threads, lb, st);
}

cudaError_t launch_fix_x(const cfs_plan* P, const double* in, double* out, bool inverse, double mul,
                         cudaStream_t st, long long nlines) {
  if (nlines < 0) nlines = (long long)P->ny * P->nz;
  if (nlines == 0) return cudaSuccess;
  return inverse ? dispatch<true>(P, in, out, mul, nlines, st)
                 : dispatch<false>(P, in, out, mul, nlines, st);
}

}  // namespace chanfs
