// mgr_solve.cuh -- Thomas solves of the coarse mass matrix along one axis
// (arXiv 2105.12764, Sec. III.A.3) and the coarsest-grid copy, as per-CTA
// bodies (used by the single-field kernels below and by the batched ones).
//
// The LU of the coarse mass matrix is scaled so each step is one FMA (the
// diagonal 1/u_q is folded into the mass-transfer stencil):
//   forward   y_q = f'_q - ta_q * y_{q-1}
//   backward  z_q = y_q  - tb_q * z_{q+1}
// The last axis of a level applies the correction (Eq. (1)) into the coarse
// workspace: w += z (decompose) or w -= z (recompose).
#pragma once

enum { SOLVE_INPLACE = 0, SOLVE_ADD = 1, SOLVE_SUB = 2 };

template <typename TW>
__device__ __forceinline__ void apply_op(TW* f, TW* w, int64_t g, TW v, int op) {
  if (op == SOLVE_INPLACE) f[g] = v;
  else if (op == SOLVE_ADD) w[g] = w[g] + v;
  else w[g] = w[g] - v;
}

// Lines along a strided axis, one thread per line: element q of line
// (o, i) sits at o*ostride + i + q*lstride; consecutive threads take
// consecutive i, so every step is a coalesced access.  `line` is this
// thread's line index in [0, inner*outer).  The recurrence runs through U
// elements at a time.  AHEAD: the next U are loaded before the recurrence runs
// (a load written after a step's store would wait for it): the single-field
// solves, whose few warps per SM otherwise alternate between waiting for loads
// and running recurrences (513^3 FP64: y 0.105 -> 0.094 ms, z 0.144 -> 0.118;
// 1000x700x300, FP64 solves: z 0.250 -> 0.195; 2049 x 3000 FP32: y 0.138 -> 0.095).
// The batched solves have enough warps without it (1024 fields: z 0.130 ms, 0.184
// with it).
template <typename TW, int U, bool AHEAD>
__device__ __forceinline__ void solve_strided_line(TW* __restrict__ f, TW* __restrict__ w, int mline, int64_t lstride,
                                                   int inner, int64_t ostride, const TW* __restrict__ ta,
                                                   const TW* __restrict__ tb, int op, int64_t line,
                                                   long long ext = 0) {
  (void)ext;  // elements of f and w (the coarse grid): checked in bounds-checking builds
  const int i = int(line % inner);
  const int64_t o = line / inner;
  // the line's elements are o*ostride + i + q*lstride, q = 0..mline-1: its ends bound them all
  if (!MGR_IN(o * ostride + i, ext, kDbgSolveF) || !MGR_IN(o * ostride + i + int64_t(mline - 1) * lstride, ext, kDbgSolveF))
    return;
  TW* fl = f + o * ostride + i;
  TW* wl = w + o * ostride + i;
  const bool add = op != SOLVE_INPLACE;
  TW cur[U], nxt[U], curw[U], nxtw[U];
  // elements q0 .. q0+U-1 (forward) and q1 .. q1-U+1 (backward, with those of w);
  // ALL: none of them lies outside the line
  auto up = [&](auto all, TW(&v)[U], int q0) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (all.value || q0 + u < mline) v[u] = fl[int64_t(q0 + u) * lstride];
  };
  auto down = [&](auto all, TW(&v)[U], TW(&vw)[U], int q1) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (all.value || q1 - u >= 0) {
        v[u] = fl[int64_t(q1 - u) * lstride];
        if (add) vw[u] = wl[int64_t(q1 - u) * lstride];
      }
  };
  TW prev = TW(0), next = TW(0);
  auto forward = [&](auto all, int q0) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (all.value || q0 + u < mline) {
        prev = cur[u] - ta[q0 + u] * prev;
        fl[int64_t(q0 + u) * lstride] = prev;
      }
  };
  auto backward = [&](auto all, int q1) {
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (all.value || q1 - u >= 0) {
        const int q = q1 - u;
        next = cur[u] - tb[q] * next;
        if (op == SOLVE_INPLACE) fl[int64_t(q) * lstride] = next;
        else if (op == SOLVE_ADD) wl[int64_t(q) * lstride] = curw[u] + next;
        else wl[int64_t(q) * lstride] = curw[u] - next;
      }
  };
  using Yes = std::true_type;
  using No = std::false_type;
  if constexpr (AHEAD) {
    up(No{}, cur, 0);
    int q0 = 0;
    for (; q0 + 2 * U <= mline; q0 += U) {
      up(Yes{}, nxt, q0 + U);
      forward(Yes{}, q0);
#pragma unroll
      for (int u = 0; u < U; ++u) cur[u] = nxt[u];
    }
    for (; q0 < mline; q0 += U) {
      up(No{}, nxt, q0 + U);
      forward(No{}, q0);
#pragma unroll
      for (int u = 0; u < U; ++u) cur[u] = nxt[u];
    }
    down(No{}, cur, curw, mline - 1);
    int q1 = mline - 1;
    for (; q1 >= 2 * U - 1; q1 -= U) {
      down(Yes{}, nxt, nxtw, q1 - U);
      backward(Yes{}, q1);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        cur[u] = nxt[u];
        curw[u] = nxtw[u];
      }
    }
    for (; q1 >= 0; q1 -= U) {
      down(No{}, nxt, nxtw, q1 - U);
      backward(No{}, q1);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        cur[u] = nxt[u];
        curw[u] = nxtw[u];
      }
    }
  } else {
    for (int q0 = 0; q0 < mline; q0 += U) {
      up(No{}, cur, q0);
      forward(No{}, q0);
    }
    for (int q1 = mline - 1; q1 >= 0; q1 -= U) {
      down(No{}, cur, curw, q1);
      backward(No{}, q1);
    }
  }
}

#ifndef MGR_SOLVE_U32
#define MGR_SOLVE_U32 16
#endif
#ifndef MGR_SOLVE_U64
#define MGR_SOLVE_U64 8
#endif
// One warp per CTA: the warps of a level's lines (2064 at 257^3) then spread over
// the SMs one by one.
constexpr int kStridedThreads = 32;
template <typename TW>
__global__ void __launch_bounds__(kStridedThreads) k_solve_strided(TW* __restrict__ f, TW* __restrict__ w, int mline,
                                                       int64_t lstride, int inner, int64_t outer, int64_t ostride,
                                                       const TW* __restrict__ ta, const TW* __restrict__ tb, int op) {
  const int64_t id = blockIdx.x * int64_t(blockDim.x) + threadIdx.x;
  if (id >= int64_t(inner) * outer) return;
  solve_strided_line<TW, sizeof(TW) == 4 ? MGR_SOLVE_U32 : MGR_SOLVE_U64, true>(f, w, mline, lstride, inner, ostride, ta, tb, op, id,
                                                   max(int64_t(mline) * lstride, outer * ostride));
}

// Lines along a strided axis, NL (32, 16 or 8) per CTA, staged whole in shared
// memory: the CTA's lines (consecutive line indices, so each step q is one or two
// contiguous row segments) are copied in with asynchronous copies all in
// flight, NL threads run the recurrences on the staged lines, and the CTA
// writes them back (or applies the correction).  Each element crosses HBM
// once each way instead of twice, and all of a CTA's loads are in flight at
// once: the form for coarse levels and planes, whose few lines leave the
// one-thread-per-line kernel latency-bound.  With many lines the single computing
// warp per CTA bounds it, and the one-thread-per-line kernel is faster.  Fewer
// lines per CTA spread few lines over the SMs and let long ones fit (2049 x 3000,
// 1501 lines of 1025, y: FP32 one thread per line 0.090 ms, staged 0.035; FP64
// 0.232, staged 0.094).  The stores of a batch follow its recurrence: between its
// steps they held up the next one (257^3 FP64, 16641 lines of 129: 31 -> 20 us).
constexpr int kStagedThreads = 256;

template <typename TW>
size_t solve_staged_smem(int mline, int nl) {
  return sizeof(TW) * (size_t(mline) * nl + 2 * size_t(mline)) + sizeof(int64_t) * nl;
}

template <typename TW, int NL>
__global__ void __launch_bounds__(kStagedThreads) k_solve_staged(TW* __restrict__ f, TW* __restrict__ w, int mline,
                                                                 int64_t lstride, int inner, int64_t outer,
                                                                 int64_t ostride, const TW* __restrict__ ta,
                                                                 const TW* __restrict__ tb, int op) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int64_t l0 = int64_t(blockIdx.x) * NL;
  int64_t* off = reinterpret_cast<int64_t*>(smem_raw);  // [NL] offset of each line's first element
  TW* s = reinterpret_cast<TW*>(off + NL);                 // [mline][NL]
  TW* sa = s + int64_t(mline) * NL;                        // [mline]
  TW* sb = sa + mline;                                     // [mline]
  const int64_t lines = int64_t(inner) * outer;
  const int nl = int(lines - l0 < NL ? lines - l0 : NL);
  if (threadIdx.x < NL) {
    const int64_t line = l0 + (threadIdx.x < nl ? threadIdx.x : 0);
    const int64_t o = line / inner;
    const int64_t first = o * ostride + (line - o * inner);
#ifdef MGR_DEBUG_BOUNDS
    // a line's elements are first + q*lstride: its ends bound them all (out of
    // bounds: recorded, and the line is pointed at element 0 to stay inside)
    const long long ext = max(int64_t(mline) * lstride, outer * ostride);
    const bool ok = MGR_IN(first, ext, kDbgSolveF) && MGR_IN(first + int64_t(mline - 1) * lstride, ext, kDbgSolveF);
    off[threadIdx.x] = ok ? first : 0;
#else
    off[threadIdx.x] = first;
#endif
  }
  for (int q = threadIdx.x; q < mline; q += kStagedThreads) {
    sa[q] = ta[q];
    sb[q] = tb[q];
  }
  __syncthreads();
  // a thread's line is the same in every step of its loops
  const int total = mline * NL, j = threadIdx.x % NL, q0 = threadIdx.x / NL;
  constexpr int dq = kStagedThreads / NL;
  const int64_t step = dq * lstride;
  if (j < nl) {
    const TW* src = f + off[j] + q0 * lstride;
    for (int e = threadIdx.x; e < total; e += kStagedThreads, src += step) cp_async(s + e, src, int(sizeof(TW)));
  }
  cp_commit();
  cp_wait<0>();
  __syncthreads();
  if (threadIdx.x < nl) {
    // U elements at a time, the next U loaded ahead of the stores
    constexpr int U = 8;
    TW* l = s + threadIdx.x;
    TW v[U], a[U], vn[U], an[U];
    auto up = [&](TW(&x)[U], TW(&c)[U], int q) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int qq = min(q + u, mline - 1);
        x[u] = l[qq * NL];
        c[u] = sa[qq];
      }
    };
    TW prev = TW(0);
    up(v, a, 0);
    for (int q = 0; q < mline; q += U) {
      up(vn, an, q + U);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        prev = v[u] - a[u] * prev;
        v[u] = prev;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (q + u < mline) l[(q + u) * NL] = v[u];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        v[u] = vn[u];
        a[u] = an[u];
      }
    }
    auto down = [&](TW(&x)[U], TW(&c)[U], int q) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int qq = max(q - u, 0);
        x[u] = l[qq * NL];
        c[u] = sb[qq];
      }
    };
    TW next = TW(0);
    down(v, a, mline - 1);
    for (int q = mline - 1; q >= 0; q -= U) {
      down(vn, an, q - U);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        next = v[u] - a[u] * next;
        v[u] = next;
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (q - u >= 0) l[(q - u) * NL] = v[u];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        v[u] = vn[u];
        a[u] = an[u];
      }
    }
  }
  __syncthreads();
  if (j >= nl) return;
  constexpr int W = 8;
  TW* fo = f + off[j] + q0 * lstride;
  TW* wo = w + off[j] + q0 * lstride;
  for (int e0 = threadIdx.x; e0 < total; e0 += W * kStagedThreads) {
    TW sv[W], wv[W];
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int e = e0 + u * kStagedThreads;
      sv[u] = e < total ? s[e] : TW(0);
      wv[u] = (op != SOLVE_INPLACE && e < total) ? wo[u * step] : TW(0);
    }
#pragma unroll
    for (int u = 0; u < W; ++u) {
      if (e0 + u * kStagedThreads >= total) break;
      if (op == SOLVE_INPLACE) fo[u * step] = sv[u];
      else if (op == SOLVE_ADD) wo[u * step] = wv[u] + sv[u];
      else wo[u * step] = wv[u] - sv[u];
    }
    fo += W * step;
    wo += W * step;
  }
}

// Lines along the contiguous axis: R rows of length mline (one after another)
// starting at row r0 are staged in shared memory with coalesced
// asynchronous copies by all threads; thread r < R then runs its row's
// recurrences through 16-byte vectors of the staged row (one shared load,
// E = 16 / sizeof(TW) dependent FMAs and one shared store per vector), and
// all threads write the rows back.  The recurrence coefficients are staged
// once, zero-padded to the pitch.
//
// Shared row pitch: a whole, odd number of 16-byte vectors.  A 16-byte shared
// access is served eight threads at a time, and rows whose starts differ by
// an odd number of vectors put those eight in different bank groups.
template <typename TW>
constexpr int contig_pitch(int mline) {
  constexpr int E = 16 / int(sizeof(TW));
  const int v = (mline + E - 1) / E;
  return ((v & 1) ? v : v + 1) * E;
}
template <typename TW>
constexpr size_t solve_contig_smem(int mline, int R) {
  return sizeof(TW) * (size_t(R) + 2) * size_t(contig_pitch<TW>(mline));
}
template <typename TW>
struct Vec16;
template <>
struct Vec16<float> {
  using type = float4;
};
template <>
struct Vec16<double> {
  using type = double2;
};

template <typename TW>
__device__ __forceinline__ void solve_contig_rows(TW* __restrict__ f, TW* __restrict__ w, int mline, int64_t rows, int R,
                                                  const TW* __restrict__ ta,
                                                  const TW* __restrict__ tb, int op, int64_t r0,
                                                  unsigned char* smem_raw) {
  const int pitch = contig_pitch<TW>(mline);
  TW* s = reinterpret_cast<TW*>(smem_raw);  // [R][pitch]
  TW* sa = s + R * pitch;                   // [pitch], zero past mline
  TW* sb = sa + pitch;                      // [pitch], zero past mline
  const int nr = int(rows - r0 < int64_t(R) ? rows - r0 : int64_t(R));
  // rows r0 .. r0+nr-1 of mline elements
  if (!MGR_IN((r0 + nr) * mline - 1, rows * mline, kDbgSolveF)) return;
  // The rows lie one after another: they go to shared memory
  // as element-wise asynchronous copies, all in flight at once, thread by thread
  // over the whole block of elements, whatever the row length (a warp per row
  // left 31 of 32 lanes idle on the last element of a row of 33).
  const int total = nr * mline, nt = blockDim.x;
  const int dr = nt / mline, dc = nt - dr * mline;  // rows and columns per step of nt elements
  const int er = threadIdx.x / mline, ec = threadIdx.x - er * mline;
  const TW* src = f + r0 * mline;
  for (int e = threadIdx.x, r = er, c = ec; e < total; e += nt) {
    cp_async(s + r * pitch + c, src + e, int(sizeof(TW)));
    r += dr;
    c += dc;
    if (c >= mline) {
      c -= mline;
      ++r;
    }
  }
  cp_commit();
  for (int q = threadIdx.x; q < pitch; q += blockDim.x) {
    sa[q] = q < mline ? ta[q] : TW(0);
    sb[q] = q < mline ? tb[q] : TW(0);
  }
  cp_wait<0>();
  __syncthreads();
  if (threadIdx.x < nr) {
    using V = typename Vec16<TW>::type;
    constexpr int E = 16 / int(sizeof(TW));
    V* l = reinterpret_cast<V*>(s + threadIdx.x * pitch);
    const V* av = reinterpret_cast<const V*>(sa);
    const V* bv = reinterpret_cast<const V*>(sb);
    const int nv = (mline + E - 1) / E;  // vectors holding the row's elements
    // forward: the elements past mline in the last vector follow every real
    // one, so computing on them (the padding) changes nothing that is kept
    // (the next two vectors are loaded ahead of each store: a load written after
    // it would wait for it; 2049 x 3000 FP64: 0.149 -> 0.132 ms)
    TW prev = TW(0);
    V xn = l[0], an = av[0], xm = l[min(1, nv - 1)], am = av[min(1, nv - 1)];
#pragma unroll 2
    for (int i = 0; i < nv; ++i) {
      alignas(16) TW x[E];
      alignas(16) TW a[E];
      *reinterpret_cast<V*>(x) = xn;
      *reinterpret_cast<V*>(a) = an;
      xn = xm;
      an = am;
      const int j = min(i + 2, nv - 1);
      xm = l[j];
      am = av[j];
#pragma unroll
      for (int e = 0; e < E; ++e) {
        prev = x[e] - a[e] * prev;
        x[e] = prev;
      }
      l[i] = *reinterpret_cast<const V*>(x);
    }
    // backward from element mline-1: in the last vector the elements past
    // mline are skipped
    TW next = TW(0);
    {
      const int i = nv - 1;
      alignas(16) TW x[E];
      alignas(16) TW b[E];
      *reinterpret_cast<V*>(x) = l[i];
      *reinterpret_cast<V*>(b) = bv[i];
#pragma unroll
      for (int e = E - 1; e >= 0; --e)
        if (i * E + e < mline) {
          next = x[e] - b[e] * next;
          x[e] = next;
        }
      l[i] = *reinterpret_cast<const V*>(x);
    }
    V yn = l[max(nv - 2, 0)], bn = bv[max(nv - 2, 0)], ym = l[max(nv - 3, 0)], bm = bv[max(nv - 3, 0)];
#pragma unroll 2
    for (int i = nv - 2; i >= 0; --i) {
      alignas(16) TW x[E];
      alignas(16) TW b[E];
      *reinterpret_cast<V*>(x) = yn;
      *reinterpret_cast<V*>(b) = bn;
      yn = ym;
      bn = bm;
      const int j = max(i - 2, 0);
      ym = l[j];
      bm = bv[j];
#pragma unroll
      for (int e = E - 1; e >= 0; --e) {
        next = x[e] - b[e] * next;
        x[e] = next;
      }
      l[i] = *reinterpret_cast<const V*>(x);
    }
  }
  __syncthreads();
  // write back (or apply the correction to w) in the same order, W elements per
  // thread per round with their loads of w issued together
  constexpr int W = 4;
  TW* fo = f + r0 * mline;
  TW* wo = w + r0 * mline;
  for (int e0 = threadIdx.x, r = er, c = ec; e0 < total; e0 += W * nt) {
    TW sv[W], wv[W];
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int e = e0 + u * nt;
      sv[u] = e < total ? s[r * pitch + c] : TW(0);
      wv[u] = (op != SOLVE_INPLACE && e < total) ? wo[e] : TW(0);
      r += dr;
      c += dc;
      if (c >= mline) {
        c -= mline;
        ++r;
      }
    }
#pragma unroll
    for (int u = 0; u < W; ++u) {
      const int e = e0 + u * nt;
      if (e >= total) break;
      if (op == SOLVE_INPLACE) fo[e] = sv[u];
      else if (op == SOLVE_ADD) wo[e] = wv[u] + sv[u];
      else wo[e] = wv[u] - sv[u];
    }
  }
}

template <typename TW>
__global__ void __launch_bounds__(128) k_solve_contig(TW* __restrict__ f, TW* __restrict__ w, int mline, int64_t rows, int R,
                                                      const TW* __restrict__ ta,
                                                      const TW* __restrict__ tb, int op) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  solve_contig_rows<TW>(f, w, mline, rows, R, ta, tb, op, blockIdx.x * int64_t(R), smem_raw);
}

// Lines along the contiguous axis, 32 per warp (lane = line): the warp moves
// its lines through a 32 x 32 shared-memory tile (row segments loaded and
// stored coalesced, transposed in the tile), each lane runs its line's
// recurrence through the tile's columns.  The forward sweep writes y back to
// f, the backward sweep reads it again; no whole line is held on chip, so
// many warps (hence many independent recurrences) fit on an SM.
constexpr int kRowsWarps = 4;

template <typename TW>
__global__ void __launch_bounds__(kRowsWarps * 32) k_solve_rows(TW* __restrict__ f, TW* __restrict__ w, int mline,
                                                                int64_t rows, int64_t row_pitch,
                                                                const TW* __restrict__ ta, const TW* __restrict__ tb,
                                                                int op) {
  // loads of a tile are issued in batches of B before their shared-memory
  // stores (128 bytes of loads in flight per thread)
  constexpr int B = 128 / sizeof(TW);
  __shared__ TW tiles[kRowsWarps][32][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t r0 = (int64_t(blockIdx.x) * kRowsWarps + warp) * 32;
  if (r0 >= rows) return;
  const int nr = int(rows - r0 < 32 ? rows - r0 : 32);
  // rows r0 .. r0+nr-1 of mline elements at pitch row_pitch
  if (!MGR_IN((r0 + nr - 1) * row_pitch + mline - 1, rows * row_pitch, kDbgSolveF)) return;
  TW(*tile)[33] = tiles[warp];
  TW* base = f + r0 * row_pitch;
  TW* wb = w + r0 * row_pitch;
  const bool act = lane < nr;
  auto load_tile = [&](int c0) {
#pragma unroll
    for (int i0 = 0; i0 < 32; i0 += B) {
      TW v[B];
#pragma unroll
      for (int u = 0; u < B; ++u) v[u] = (i0 + u < nr) ? base[int64_t(i0 + u) * row_pitch + c0 + lane] : TW(0);
#pragma unroll
      for (int u = 0; u < B; ++u) tile[lane][i0 + u] = v[u];
    }
  };
  TW prev = TW(0);
  for (int c0 = 0; c0 < mline; c0 += 32) {
    const int nc = min(32, mline - c0);
    if (lane < nc) load_tile(c0);
    __syncwarp();
    if (act) {
      for (int c = 0; c < nc; c += 8) {
        TW v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = tile[c + u][lane];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (c + u < nc) prev = v[u] - ta[c0 + c + u] * prev;
          v[u] = prev;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) tile[c + u][lane] = v[u];
      }
    }
    __syncwarp();
    if (lane < nc) {
#pragma unroll 8
      for (int i = 0; i < nr; ++i) base[int64_t(i) * row_pitch + c0 + lane] = tile[lane][i];
    }
    __syncwarp();
  }
  TW next = TW(0);
  for (int c0 = ((mline - 1) / 32) * 32; c0 >= 0; c0 -= 32) {
    const int nc = min(32, mline - c0);
    if (lane < nc) load_tile(c0);
    __syncwarp();
    if (act) {
      for (int c = (nc - 1) & ~7; c >= 0; c -= 8) {
        TW v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = tile[c + u][lane];
#pragma unroll
        for (int u = 7; u >= 0; --u) {
          if (c + u < nc) next = v[u] - tb[c0 + c + u] * next;
          v[u] = next;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) tile[c + u][lane] = v[u];
      }
    }
    __syncwarp();
    if (lane < nc) {
      if (op == SOLVE_INPLACE) {
#pragma unroll 8
        for (int i = 0; i < nr; ++i) base[int64_t(i) * row_pitch + c0 + lane] = tile[lane][i];
      } else {
        const TW sg = op == SOLVE_ADD ? TW(1) : TW(-1);
#pragma unroll
        for (int i0 = 0; i0 < 32; i0 += B) {
          TW v[B];
#pragma unroll
          for (int u = 0; u < B; ++u) v[u] = (i0 + u < nr) ? wb[int64_t(i0 + u) * row_pitch + c0 + lane] : TW(0);
#pragma unroll
          for (int u = 0; u < B; ++u)
            if (i0 + u < nr) wb[int64_t(i0 + u) * row_pitch + c0 + lane] = v[u] + sg * tile[lane][i0 + u];
        }
      }
    }
    __syncwarp();
  }
}

// Coarsest grid <-> nodal positions (dir 0: gather nodal -> compact; 1: scatter)
template <typename TD, typename TW>
__device__ __forceinline__ void coarsest_copy(TD* y, int64_t y_sz, int64_t y_sy, TW* w, int3 n, longlong3 s,
                                              longlong3 N, int dir, int64_t e0, int64_t estep) {
  const int64_t total = int64_t(n.x) * n.y * n.z;
  for (int64_t e = e0; e < total; e += estep) {
    const int gx = int(e % n.z);
    const int64_t rest = e / n.z;
    const int gy = int(rest % n.y), gz = int(rest / n.y);
    const int64_t yo = fmap(gz, s.x, N.x) * y_sz + fmap(gy, s.y, N.y) * y_sy + fmap(gx, s.z, N.z);
    if (!MGR_IN(yo, N.x * y_sz, kDbgCoarsestY)) continue;
    if (dir == 0) w[e] = TW(y[yo]);
    else y[yo] = TD(w[e]);
  }
}

template <typename TD, typename TW>
__global__ void k_coarsest(TD* y, int64_t y_sz, int64_t y_sy, TW* w, int3 n, longlong3 s, longlong3 N, int dir) {
  coarsest_copy<TD, TW>(y, y_sz, y_sy, w, n, s, N, dir, blockIdx.x * int64_t(blockDim.x) + threadIdx.x,
                        int64_t(gridDim.x) * blockDim.x);
}
