// FP32 product on the orbital factorisation of a block pair (Sec. 2.4: inside
// a block H_sigma is a Kronecker sum over the orbital groups).
//
// The columns of an up block are the mixed-radix numbers of its group strings
// (group 0 slowest), so a row of the block is a tensor [L_0][L_1]..[L_m-1],
// L_k = C(G, n_k), and the hops of orbital k act along axis k alone, with the
// sign of the other groups' occupations the same for every element of a
// fibre of that axis.  Which elements of a fibre a hop connects, with which
// bath level and which sign inside the group, depends on (G, n_k) only, so
// it is compiled in: a thread loads a fibre (at most 70 elements) into
// registers and forms all its hops with straight-line FMAs whose matrix
// elements sit in G - 1 registers.  No index or value table is read, each
// element is loaded once per axis and each accumulator loaded and stored
// once.
//
// Order of the terms per element: the diagonal, the hops of groups 0..m-2 in
// ascending target index, the hops of the last group, the H_dw terms in CSR
// order: the order of the ELL entries, so w equals the element-parallel
// product bit for bit.  Levels inside a group are the impurity (bit 0) and
// its bath levels, so a hop out of an impurity-empty string lowers the index
// and one out of an occupied string raises it: ascending targets are the
// impurity-empty halves of axes 0, 1, .. m-2, then the occupied halves of
// axes m-2, .. 0.
//
// Bound: shared-memory wavefronts (about 14 words per element: staging, two or
// three accesses per axis, output) and the barriers between the axes; without
// its axes the pass moves v and w at 5.8 TB/s.  Measured (GB300, whole H_up
// pass): three orbitals at Ns = 18 17.4 -> 7.5 ms, two orbitals at Ns = 16
// 0.49 ms, against kernels that read an ELL table of H_up from L2 and gather
// staged rows.  Tried and slower: persistent CTAs that prefetch the next item
// (8.2 / 0.53 ms: fewer warps per SM), pairs of rows on packed FP32 FMAs (7.7 /
// 0.57 ms: half the instructions, half the warps), halves of the 70-element
// fibres on separate threads (0.65 ms), E_up staged with the rows (8.4 ms).
#pragma once

#include <utility>

#include "product.cuh"

namespace fiber {

constexpr int binom(int n, int k) {
  if (k < 0 || k > n) return 0;
  long long r = 1;
  for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
  return (int)r;
}
constexpr int popc(unsigned x) {
  int c = 0;
  for (; x; x &= x - 1) ++c;
  return c;
}
// i-th string of n bits in ascending order, and its rank
constexpr unsigned nth_string(int n, int i) {
  unsigned s = 0;
  for (int k = n; k >= 1; --k) {
    int p = k - 1;
    while (binom(p + 1, k) <= i) ++p;
    i -= binom(p, k);
    s |= 1u << p;
  }
  return s;
}
constexpr int string_rank(unsigned s) {
  int r = 0, k = 0;
  for (int p = 0; p < 32; ++p)
    if ((s >> p) & 1u) r += binom(p, ++k);
  return r;
}

// Hops into element I of a group of G levels with N electrons, in ascending
// order of their source: from an impurity-empty string the occupied bath
// levels descending, from an occupied one the empty bath levels ascending.
template <int G, int N, int I>
struct Row {
  static constexpr unsigned str = nth_string(N, I);
  static constexpr bool occ = (str & 1u) != 0;
  static constexpr int cnt = occ ? G - N : N;
  static constexpr int level(int k) {  // bath level 0 .. G-2 of hop k
    if (occ) {
      for (int b = 1; b < G; ++b)
        if (!((str >> b) & 1u) && k-- == 0) return b - 1;
    } else {
      for (int b = G - 1; b >= 1; --b)
        if (((str >> b) & 1u) && k-- == 0) return b - 1;
    }
    return 0;
  }
  static constexpr int src(int k) { return string_rank(str ^ 1u ^ (2u << level(k))); }
  // sign of the occupied bath levels below the hop's
  static constexpr bool neg(int k) { return popc(str & ((2u << level(k)) - 1u) & ~1u) & 1; }
};

template <class F, int... I>
__device__ __forceinline__ void unroll_impl(std::integer_sequence<int, I...>, F &&f) {
  (f(std::integral_constant<int, I>{}), ...);
}
template <int N, class F>
__device__ __forceinline__ void unroll(F &&f) {
  unroll_impl(std::make_integer_sequence<int, N>{}, f);
}

template <int G, int N, int I, typename T, int L>
__device__ __forceinline__ T hops(const T (&x)[L], const T (&V)[G - 1], T acc) {
  using R = Row<G, N, I>;
  unroll<R::cnt>([&](auto K) {
    constexpr int k = decltype(K)::value;
    constexpr int l = R::level(k), s = R::src(k);
    constexpr bool neg = R::neg(k);
    acc = fma_t<T>(neg ? -V[l] : V[l], x[s], acc);
  });
  return acc;
}

// Accumulators are handled FIBER_CHUNK at a time, all loads of a chunk before
// its stores: the compiler has to assume that a store may change the next
// accumulator, so a load - add - store sequence per element would wait out a
// shared-memory latency for every element.
constexpr int FIBER_CHUNK = 8;

// The multiples of S are formed anew for every chunk of a long fibre: kept
// from its loads for its stores they would take a register per element (the
// 70-element fibres spilled 2 KB per thread).
template <int L>
__device__ __forceinline__ int fresh(int s) {
  if (L > 20) asm volatile("" : "+r"(s)::"memory");
  return s;
}

// The elements of (G, N) that are impurity-empty (HALF 0), occupied (1), all (2).
template <int G, int N, int HALF>
struct Half {
  static constexpr int L = binom(G, N);
  static constexpr int size = HALF == 2 ? L : (HALF == 0 ? binom(G - 1, N) : binom(G - 1, N - 1));
  static constexpr int index(int k) {
    for (int i = 0; i < L; ++i)
      if (HALF == 2 || (int)(nth_string(N, i) & 1u) == HALF)
        if (k-- == 0) return i;
    return 0;
  }
};

template <int G, int N, int HALF, typename T, int L>
__device__ __forceinline__ void load_half(const T *X, int S, T (&x)[L]) {
  using In = Half<G, N, HALF>;
  unroll<In::size>([&](auto K) {
    constexpr int i = In::index(decltype(K)::value);
    x[i] = X[i * S];
  });
}

// First axis: acc = diagonal * x, then the hops of its impurity-empty half
// (with BOTH also of the occupied half).  eu, ed, w0, w1: the diagonal's
// pieces (W at an empty and an occupied impurity level of this group).
template <int G, int N, bool BOTH, typename T>
__device__ __forceinline__ void step_first(const T *X, T *A, int S, const T (&V)[G - 1],
                                           const T *eu, T ed, T w0, T w1) {
  constexpr int L = binom(G, N);
  T x[L];
  load_half<G, N, 2, T, L>(X, S, x);
  unroll<(L + FIBER_CHUNK - 1) / FIBER_CHUNK>([&](auto C) {
    constexpr int i0 = decltype(C)::value * FIBER_CHUNK;
    constexpr int n = L - i0 < FIBER_CHUNK ? L - i0 : FIBER_CHUNK;
    T acc[n];
    const int S2 = fresh<L>(S);
    unroll<n>([&](auto Q) {
      acc[decltype(Q)::value] = __ldg(eu + (i0 + decltype(Q)::value) * S2);
    });
    unroll<n>([&](auto Q) {
      constexpr int q = decltype(Q)::value, i = i0 + q;
      using R = Row<G, N, i>;
      acc[q] = mul_t<T>(add_t<T>(add_t<T>(acc[q], ed), R::occ ? w1 : w0), x[i]);
      if constexpr (!R::occ || BOTH) acc[q] = hops<G, N, i, T, L>(x, V, acc[q]);
    });
    unroll<n>([&](auto Q) { A[(i0 + decltype(Q)::value) * S2] = acc[decltype(Q)::value]; });
  });
}

// An inner axis: WHICH 0 the impurity-empty outputs, 1 the occupied ones, 2 both.
template <int G, int N, int WHICH, typename T>
__device__ __forceinline__ void step_mid(const T *X, T *A, int S, const T (&V)[G - 1]) {
  constexpr int L = binom(G, N);
  using Out = Half<G, N, WHICH>;
  T x[L];
  load_half<G, N, WHICH == 2 ? 2 : 1 - WHICH, T, L>(X, S, x);
  unroll<(Out::size + FIBER_CHUNK - 1) / FIBER_CHUNK>([&](auto C) {
    constexpr int k0 = decltype(C)::value * FIBER_CHUNK;
    constexpr int n = Out::size - k0 < FIBER_CHUNK ? Out::size - k0 : FIBER_CHUNK;
    T acc[n];
    const int S2 = fresh<L>(S);
    unroll<n>([&](auto Q) {
      constexpr int i = Out::index(k0 + decltype(Q)::value);
      acc[decltype(Q)::value] = A[i * S2];
    });
    unroll<n>([&](auto Q) {
      constexpr int q = decltype(Q)::value, i = Out::index(k0 + q);
      acc[q] = hops<G, N, i, T, L>(x, V, acc[q]);
    });
    unroll<n>([&](auto Q) {
      constexpr int i = Out::index(k0 + decltype(Q)::value);
      A[i * S2] = acc[decltype(Q)::value];
    });
  });
}

template <int W>
struct VecT;
template <>
struct VecT<1> { using type = float; };
template <>
struct VecT<2> { using type = float2; };
template <>
struct VecT<4> { using type = float4; };

// The last axis: fibres are contiguous, read and written in the widest
// vectors their length allows (an odd number of vectors per fibre, mostly,
// so that the lanes of a warp hit distinct banks).
template <int G, int N>
__device__ __forceinline__ void step_last(const float *X, float *A, const float (&V)[G - 1]) {
  constexpr int L = binom(G, N);
  constexpr int W = L % 4 == 0 ? 4 : (L % 2 == 0 ? 2 : 1);
  constexpr int LV = L / W, CV = FIBER_CHUNK / W;
  using VT = typename VecT<W>::type;
  union U {
    VT v;
    float f[W];
    __device__ U() {}
  };
  float x[L];
  unroll<LV>([&](auto I) {
    constexpr int i = decltype(I)::value;
    U u;
    u.v = reinterpret_cast<const VT *>(X)[i];
    unroll<W>([&](auto Q) { x[i * W + decltype(Q)::value] = u.f[decltype(Q)::value]; });
  });
  unroll<(LV + CV - 1) / CV>([&](auto C) {
    constexpr int i0 = decltype(C)::value * CV;
    constexpr int n = LV - i0 < CV ? LV - i0 : CV;
    U u[n];
    unroll<n>([&](auto J) {
      u[decltype(J)::value].v = reinterpret_cast<const VT *>(A)[i0 + decltype(J)::value];
    });
    unroll<n>([&](auto J) {
      constexpr int j = decltype(J)::value;
      unroll<W>([&](auto Q) {
        constexpr int q = decltype(Q)::value;
        u[j].f[q] = hops<G, N, (i0 + j) * W + q, float, L>(x, V, u[j].f[q]);
      });
    });
    unroll<n>([&](auto J) {
      reinterpret_cast<VT *>(A)[i0 + decltype(J)::value] = u[decltype(J)::value].v;
    });
  });
}

// ----------------------------------------------------------------- kernel

// Shapes of a CTA: CAP elements for the rows of v and as many for the
// accumulators (at least one row of the widest block of the shape), threads
// and CTAs per SM.  A CTA alternates between waiting for its rows, the axes
// and the output rows; the other CTAs of the SM fill the waits.
template <int G, int SHAPE>
struct Shape {
  static constexpr int CAP = FIBER_CAP[SHAPE];
  static constexpr int NT = SHAPE == 1 ? 256 : (G >= 7 ? 128 : 160);
  static constexpr int CTAS = SHAPE == 1 ? 3 : (G >= 7 ? 4 : 5);
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src) : "memory");
}

enum { STEP_FIRST = 0, STEP_FIRST_BOTH, STEP_EMPTY, STEP_OCC, STEP_MID, STEP_LAST };

// i / n for 0 <= i < 2^21 with inv = 1 / n: (i + 1/2) / n lies at least
// 1 / (2 n) from an integer, more than the rounding of the product
__device__ __forceinline__ int fast_div(int i, float inv) {
  return __float2int_rz(((float)i + 0.5f) * inv);
}

// Item: rows r0 .. r0 + nr of one up block.
struct FibItem {
  int r0, nr, c0, nc, c0p, deg;
};

struct RowData {
  const float *ed;     // [rows] E_dw
  const uint8_t *md;   // [rows] impurity mask
  const float *w;      // [dw mask][up mask] W
};

template <int G, int N, int KIND, typename T>
__device__ __forceinline__ void step_n(const HvTables<T> &tb, const FibItem &it, T *X, T *A, int k,
                                       int S, int parity, const RowData &rd) {
  constexpr int L = binom(G, N);
  if constexpr (KIND >= STEP_EMPTY && (N == 0 || N == G)) return;
  const int nf = it.nc / L, total = nf * it.nr;
  const float inv_nf = 1.0f / (float)nf, inv_s = 1.0f / (float)S;
  const int pitch = (it.nc + 3) & ~3;
  const unsigned bit = 1u << k;
  for (int idx = threadIdx.x; idx < total; idx += blockDim.x) {
    const int row = fast_div(idx, inv_nf), f = idx - row * nf;
    const int hi = fast_div(f, inv_s), base = hi * (L - 1) * S + f;  // hi L S + (f - hi S)
    const unsigned others = (unsigned)__ldg(tb.m_up + it.c0 + base) & ~bit;
    const bool neg = ((__popc(others) + parity) & 1) != 0;
    T V[G - 1];
    unroll<G - 1>([&](auto I) {
      constexpr int l = decltype(I)::value;
      const T h = tb.hop_up[k * (G - 1) + l];
      V[l] = neg ? -h : h;
    });
    const T *x = X + row * pitch + base;
    T *acc = A + row * pitch + base;
    if constexpr (KIND == STEP_FIRST || KIND == STEP_FIRST_BOTH) {
      const T *w = rd.w + rd.md[row] * tb.nmask;
      step_first<G, N, KIND == STEP_FIRST_BOTH, T>(x, acc, S, V, tb.e_up + it.c0 + base,
                                                   rd.ed[row], w[others], w[others | bit]);
    } else if constexpr (KIND == STEP_LAST) {
      step_last<G, N>(x, acc, V);
    } else {
      step_mid<G, N, KIND == STEP_EMPTY ? 0 : (KIND == STEP_OCC ? 1 : 2), T>(x, acc, S, V);
    }
  }
}

template <int G, int KIND, typename T, int N = 0>
__device__ __forceinline__ void step(int n, const HvTables<T> &tb, const FibItem &it, T *X, T *A,
                                     int k, int S, int parity, const RowData &rd) {
  if (n == N) {
    step_n<G, N, KIND, T>(tb, it, X, A, k, S, parity, rd);
  } else if constexpr (N < G) {
    step<G, KIND, T, N + 1>(n, tb, it, X, A, k, S, parity, rd);
  }
}

// H_up pass: one item (rows x one up block) per CTA; the
// diagonal and H_up, written unscaled (k_hv_dw adds H_dw).  lanczos: the
// vectors of the recurrence (step j of the device state) instead of a.v, a.w.
template <int G, int SHAPE>
__global__ void __launch_bounds__(Shape<G, SHAPE>::NT, Shape<G, SHAPE>::CTAS)
    k_hv_fiber(HvLaunch<float> a, int lanczos) {
  constexpr int CAP = Shape<G, SHAPE>::CAP, NT = Shape<G, SHAPE>::NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float *const X = reinterpret_cast<float *>(smem_raw), *const A = X + CAP;
  __shared__ float s_ed[FIBER_ROWS], s_w[1 << (2 * FIBER_MAX_W_NORB)];
  __shared__ uint8_t s_md[FIBER_ROWS];
  __shared__ FibItem s_it;
  const HvTables<float> &tb = a.tb;
  const float *g = a.v + blockIdx.y * a.slice;
  float *out = a.w + blockIdx.y * a.slice;
  if (lanczos) {
    const LanczosState *st = a.st;
    if (st->done) return;
    const int j = st->j, m3 = j % 3;
    g = m3 == 0 ? a.b0 : (m3 == 1 ? a.b1 : a.b2);
    out = m3 == 0 ? a.b1 : (m3 == 1 ? a.b2 : a.b0);
    if (a.basis) {
      g = a.basis[j];
      out = a.basis[j + 1];
    }
  }
  // the item's up block: the last one whose first item is not above this item
  if (threadIdx.x < 32) {
    FibItem it;
    const int item = (int)(tb.fib_first[SHAPE] + blockIdx.x);
    const FibBlock *fb = tb.fib[SHAPE];
    int b = 0;
    for (int q = 0; q < tb.nfib[SHAPE]; q += 32) {
      const int lane = q + (int)(threadIdx.x & 31);
      const unsigned le =
          __ballot_sync(0xffffffffu, lane < tb.nfib[SHAPE] && fb[lane].first <= item);
      if (!le) break;
      b = q + 31 - __clz(le);
    }
    const FibBlock blk = fb[b];
    it.c0 = blk.c0;
    it.nc = blk.nc;
    it.c0p = blk.c0p;
    it.deg = blk.keys;
    const int64_t r = (int64_t)(item - blk.first) * blk.rows;
    it.r0 = (int)(tb.row0 + r);
    it.nr = (int)min((int64_t)blk.rows, tb.rows - r);
    if (threadIdx.x == 0) s_it = it;
  }
  __syncthreads();
  const FibItem &it = s_it;
  const int64_t stride = tb.stride;
  const int m = tb.nd_norb, nr = it.nr, nc = it.nc, pitch = (nc + 3) & ~3;
  g += (int64_t)it.r0 * stride + it.c0p;
  out += (int64_t)it.r0 * stride + it.c0p;
  const int nv = pitch / 4, total = nv * nr;
  const float inv_nv = 1.0f / (float)nv;
  // the rows of v (padding columns ride along, never used)
  for (int i = threadIdx.x; i < total; i += NT) {
    const int row = fast_div(i, inv_nv), c = (i - row * nv) * 4;
    cp_async16(X + i * 4, g + (int64_t)row * stride + c);
  }
  for (int i = threadIdx.x; i < tb.nmask * tb.nmask; i += NT)
    s_w[i] = tb.W[(i % tb.nmask) * tb.nmask + i / tb.nmask];
  for (int row = threadIdx.x; row < nr; row += NT) {
    s_ed[row] = tb.e_dw[it.r0 + row];
    s_md[row] = tb.m_dw[it.r0 + row];
  }
  // group occupations (4 bits each), axis strides, electrons before group k
  int n[ED_MAX_NORB], S[ED_MAX_NORB], before[ED_MAX_NORB];
  {
    int b = 0;
#pragma unroll
    for (int k = 0; k < ED_MAX_NORB; ++k) {
      n[k] = k < m ? (it.deg >> (4 * k)) & 15 : 0;
      before[k] = b;
      b += n[k];
    }
    int s = 1;
#pragma unroll
    for (int k = ED_MAX_NORB - 1; k >= 0; --k) {
      S[k] = s;
      if (k < m) s *= (int)c_binom[G][n[k]];
    }
  }
  const RowData rd{s_ed, s_md, s_w};
  cp_async_wait_all();
  __syncthreads();
  if (m == 2) {
    step<G, STEP_FIRST_BOTH, float>(n[0], tb, it, X, A, 0, S[0], before[0], rd);
  } else {
    step<G, STEP_FIRST, float>(n[0], tb, it, X, A, 0, S[0], before[0], rd);
    // axes 1 .. m-2 empty halves ascending (the last of them both halves),
    // then occupied halves descending to axis 0
#pragma unroll
    for (int k = 1; k < ED_MAX_NORB - 2; ++k) {
      if (k >= m - 2) continue;
      __syncthreads();
      step<G, STEP_EMPTY, float>(n[k], tb, it, X, A, k, S[k], before[k], rd);
    }
#pragma unroll
    for (int k = ED_MAX_NORB - 2; k >= 0; --k) {
      if (k > m - 2) continue;
      __syncthreads();
      if (k == m - 2)
        step<G, STEP_MID, float>(n[k], tb, it, X, A, k, S[k], before[k], rd);
      else
        step<G, STEP_OCC, float>(n[k], tb, it, X, A, k, S[k], before[k], rd);
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 1; k < ED_MAX_NORB; ++k)
    if (k == m - 1) step<G, STEP_LAST, float>(n[k], tb, it, X, A, k, 1, before[k], rd);
  __syncthreads();

  // output rows, 4 columns per thread
  for (int q = threadIdx.x; q < total; q += NT) {
    const int row = fast_div(q, inv_nv), c = (q - row * nv) * 4;
    const float4 f = *reinterpret_cast<const float4 *>(A + q * 4);
    float *o = out + (int64_t)row * stride + c;
    if (c + 4 <= nc) {
      *reinterpret_cast<float4 *>(o) = f;
    } else {  // padding is not written
      o[0] = f.x;
      if (c + 1 < nc) o[1] = f.y;
      if (c + 2 < nc) o[2] = f.z;
    }
  }
}

template <int G, int SHAPE>
ed_status launch_one(const HvLaunch<float> *a, int mode, unsigned ns, cudaStream_t st) {
  const int64_t n = a ? a->tb.fib_n[SHAPE] : 0;
  if constexpr ((fiber_shapes(G) >> SHAPE) & 1) {
    constexpr int smem = 2 * Shape<G, SHAPE>::CAP * (int)sizeof(float);
    if (!a) {  // opt into large shared memory
      if ((mode >> SHAPE) & 1)
        ED_TRY_CUDA(cudaFuncSetAttribute(k_hv_fiber<G, SHAPE>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    } else if (n > 0) {
      k_hv_fiber<G, SHAPE><<<dim3((unsigned)n, ns), Shape<G, SHAPE>::NT, smem, st>>>(
          *a, mode == HV_LANCZOS);
      ED_LAUNCHED(1);
    }
    return ED_OK;
  }
  return n > 0 ? ED_ERR_ARG : ED_OK;
}

// One launch per shape that the sector's items need; a == nullptr: prepares
// the kernels of this G and the shapes in `mode` (bit per shape) on the current
// device.  Only those a sector has items for: an instance is a megabyte of
// code and more, which the driver loads on first use: all of them 11 ms.
template <int G>
ed_status launch_g(const HvLaunch<float> *a, int mode, unsigned ns, cudaStream_t st) {
  if (a && mode != HV_PLAIN && mode != HV_LANCZOS) return ED_ERR_ARG;
  ED_TRY((launch_one<G, 0>(a, mode, ns, st)));
  return launch_one<G, 1>(a, mode, ns, st);
}

}  // namespace fiber
