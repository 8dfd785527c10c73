// mgr_cluster.cuh -- the coarse end of the hierarchy in one thread-block cluster.
//
// Once a level grid has a few thousand to a few tens of thousand nodes, its
// level pass, line solves and interpolation are separate launches of a few
// microseconds each that leave nearly all of the chip idle.  k_coarse_dec /
// k_coarse_rec run all of those levels in one launch of kClusterSize CTAs, with the
// steps of mgr_small.cuh: every CTA owns a slab of z planes of each level, in its
// shared memory, and works on its own planes; the neighbours' planes are read, and the
// z lines exchanged, through distributed shared memory:
//
//   decompose, level l:  W = v on the own coarse nodes, A = P_2 W on the own coarse
//     planes and the next; c = v - P W; K_2, K_1 on the own planes | K_0 from own and
//     neighbouring planes, x and y solves, the own planes' part of every z line to
//     the line's owner | z solve, W + z to the owners of level l-1's planes |
//   recompose, level l:  the same from c on, W - z back to W | v = c + P W to the owners
//     of level l+1's coarse planes.
//
// (| a cluster barrier: three a level.)  The smallest levels (kLocalNodes) are done by
// every CTA for itself, without any exchange.  What bounds it is the chain of about 25
// steps of 400 to 2000 cycles, the line solves' FP64 FMAs (64 cycles each) and the barriers
// the longest.  Levels 17^3 and coarser: FP64 47 to 50 us in one CTA of 1024 threads (bound by
// the FP64 pipe of its SM: 41 thousand FMAs, 16 cycles for a warp's), 27 to 30 us here;
// FP32 25 to 27 us (bound by the issue of index arithmetic), 18 to 21 us here.
//
// A grid of one plane (2D) has its y axis where z is above, a line (1D) its x axis
// (cluster_axes).  Included inside an anonymous namespace after mgr_small.cuh.
#pragma once

constexpr int kClusterSize = 8;
// (256 threads: 33^3 FP64 69 us instead of 59; 1024: 57, but 64 registers and a whole SM each)
constexpr int kClusterThreads = 512;
// Levels of at most this many nodes every CTA does by itself, all of it: a cluster barrier
// costs 1000 cycles, a step of 9^3 nodes in one CTA 400 to 800 (with 200 here, 1025^2 FP32
// recomposes in 135 us instead of 119; with 2048 nothing changes).
constexpr size_t kLocalNodes = 1024;

// SmallArgs with the axes exchanged so that the slab axis is axis 0.
template <typename TS, typename TW>
struct ClusterArgs : SmallArgs<TS, TW> {
  int64_t st[3];  // full-grid strides of the (exchanged) axes
  int64_t total;  // elements of the full grid
  // one CTA's shared memory (byte offsets, the same in every CTA; sizes for the
  // largest slab; see cluster_layout)
  int local;                           // levels local..1 are done by every CTA alone
  int v[kSmallMaxLevels + 1];          // level l's own planes (values, coefficients)
  int w[2];                            // own coarse planes; the recomposition's levels alternate
  int f;                               // load vector of the own coarse planes
  int fz;                              // the own z lines
  int t1, t2;                          // stencil results of the own planes; t1 also A
  int tab_s[kSmallMaxLevels + 1][3];   // per level and axis: wa (n), wb (n), K (5 m)
  int tab_w[kSmallMaxLevels + 1][3];   // per level and axis: ta (m), tb (m)
};
template <typename TS, typename TW>
ClusterArgs<TS, TW> cluster_axes(const SmallArgs<TS, TW>& s) {
  ClusterArgs<TS, TW> a;
  static_cast<SmallArgs<TS, TW>&>(a) = s;
  a.st[0] = s.sz;
  a.st[1] = s.sy;
  a.st[2] = 1;
  a.total = s.N[0] * s.sz;
  const int k = s.N[0] > 1 ? 0 : s.N[1] > 1 ? 1 : 2;
  if (k == 0) return a;
  for (int l = 0; l <= kSmallMaxLevels; ++l) {
    std::swap(a.n[l][0], a.n[l][k]);
    std::swap(a.m[l][0], a.m[l][k]);
    std::swap(a.active[l][0], a.active[l][k]);
    std::swap(a.s[l][0], a.s[l][k]);
    std::swap(a.wa[l][0], a.wa[l][k]);
    std::swap(a.wb[l][0], a.wb[l][k]);
    std::swap(a.k[l][0], a.k[l][k]);
    std::swap(a.ta[l][0], a.ta[l][k]);
    std::swap(a.tb[l][0], a.tb[l][k]);
  }
  std::swap(a.N[0], a.N[k]);
  std::swap(a.s0[0], a.s0[k]);
  std::swap(a.n0[0], a.n0[k]);
  std::swap(a.st[0], a.st[k]);
  return a;
}

// Coarse planes [q0, q1) of m (rank r of the cluster), and the owner of plane q.
__host__ __device__ inline int slab_start(int r, int m) { return r * m / kClusterSize; }
__device__ __forceinline__ int slab_owner(int q, const SmallDiv& m) { return m.quo(q * kClusterSize + kClusterSize - 1); }
__host__ __device__ inline int slab_planes(int m) { return (m + kClusterSize - 1) / kClusterSize; }

// Lays a CTA's shared memory out for levels 1..a.levels; the size is the result.
template <typename TS, typename TW>
size_t cluster_layout(ClusterArgs<TS, TW>& a) {
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const int p = int(std::min(at, size_t(1) << 30));
    at += (bytes + 15) / 16 * 16;
    return p;
  };
  size_t w = 0, z = 0, t1 = 0, t2 = 0;
  a.local = 0;
  for (int l = 1; l <= a.levels; ++l) {
    const size_t n0 = a.n[l][0], n1 = a.n[l][1], n2 = a.n[l][2], m1 = a.m[l][1], m2 = a.m[l][2];
    const bool local = n0 * n1 * n2 <= kLocalNodes;
    if (local) a.local = l;
    // coarse planes and level planes of a CTA
    const size_t c = local ? a.m[l][0] : slab_planes(a.m[l][0]), i = local ? n0 : 2 * c;
    a.v[l] = take(i * n1 * n2 * sizeof(TW));
    w = std::max(w, c * m1 * m2);
    z = std::max(z, size_t(a.m[l][0]) * ((m1 * m2 + kClusterSize - 1) / kClusterSize));
    t1 = std::max(t1, std::max(i * n1 * m2, (c + 1) * m1 * n2));
    t2 = std::max(t2, i * m1 * m2);
    for (int k = 0; k < 3; ++k) {
      a.tab_s[l][k] = take((2 * size_t(a.n[l][k]) + 5 * size_t(a.m[l][k])) * sizeof(TS));
      a.tab_w[l][k] = take(2 * size_t(a.m[l][k]) * sizeof(TW));
    }
  }
  for (int& x : a.w) x = take(w * sizeof(TW));
  a.f = take(w * sizeof(TW));
  a.fz = take(z * sizeof(TW));
  a.t1 = take(t1 * sizeof(TS));
  a.t2 = take(t2 * sizeof(TS));
  return at;
}

// One level as a CTA sees it.
template <typename TS, typename TW>
struct ClusterLevel {
  int n0, n1, n2, m0, m1, m2;
  int q0, q1, i0, i1;  // own coarse planes, own level planes
  const TS *wa[3], *wb[3], *k[3];
  const TW *ta[3], *tb[3];
};
template <bool LOCAL, typename TS, typename TW>
__device__ __forceinline__ ClusterLevel<TS, TW> cluster_level(const ClusterArgs<TS, TW>& a, unsigned char* smem, int l,
                                                              int rank) {
  ClusterLevel<TS, TW> g;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int n = a.n[l][k], m = a.m[l][k];
    const TS* ts = reinterpret_cast<const TS*>(smem + a.tab_s[l][k]);
    const TW* tw = reinterpret_cast<const TW*>(smem + a.tab_w[l][k]);
    g.wa[k] = ts;
    g.wb[k] = ts + n;
    g.k[k] = ts + 2 * n;
    g.ta[k] = tw;
    g.tb[k] = tw + m;
  }
  g.n0 = a.n[l][0], g.n1 = a.n[l][1], g.n2 = a.n[l][2];
  g.m0 = a.m[l][0], g.m1 = a.m[l][1], g.m2 = a.m[l][2];
  g.q0 = LOCAL ? 0 : slab_start(rank, g.m0);
  g.q1 = LOCAL ? g.m0 : slab_start(rank + 1, g.m0);
  g.i0 = g.q0 < g.m0 ? pidx(g.q0, g.n0) : g.n0;
  g.i1 = g.q1 < g.m0 ? pidx(g.q1, g.n0) : g.n0;
  return g;
}

// Asynchronous copies of every level's tables, a table of a level and axis to a warp (the
// arguments each one needs come from a cold constant cache, 300 cycles apiece).
template <typename TS, typename TW>
__device__ __forceinline__ void cluster_copy_tables(const ClusterArgs<TS, TW>& a, unsigned char* smem) {
  auto put = [](auto* dst, const auto* src, int count) {
    for (int i = threadIdx.x & 31; i < count; i += 32) cp_async(dst + i, src + i, int(sizeof(*dst)));
  };
  for (int j = threadIdx.x >> 5; j < 15 * a.levels; j += kClusterThreads / 32) {
    const int t = j % 5, k = j / 5 % 3, l = 1 + j / 15;
    const int n = a.n[l][k], m = a.m[l][k];
    TS* s = reinterpret_cast<TS*>(smem + a.tab_s[l][k]);
    TW* w = reinterpret_cast<TW*>(smem + a.tab_w[l][k]);
    if (t == 0) put(s, a.wa[l][k], n);
    else if (t == 1) put(s + n, a.wb[l][k], n);
    else if (t == 2) put(s + 2 * n, a.k[l][k], 5 * m);
    else if (t == 3) put(w, a.ta[l][k], m);
    else put(w + m, a.tb[l][k], m);
  }
  cp_commit();
}

// The full-grid element of a level node.
template <typename TS, typename TW>
__device__ __forceinline__ int64_t cluster_full(const ClusterArgs<TS, TW>& a, const int64_t* s, int i0, int i1, int i2) {
  return fmap(i0, s[0], a.N[0]) * a.st[0] + fmap(i1, s[1], a.N[1]) * a.st[1] + fmap(i2, s[2], a.N[2]) * a.st[2];
}
template <typename T>
__device__ __forceinline__ T cluster_ld(const T* p, int64_t i, int64_t total) {
  (void)total;
  return MGR_IN(i, total, kDbgSmallIn) ? p[i] : T(0);
}
template <typename T>
__device__ __forceinline__ void cluster_st(T* p, int64_t i, T v, int64_t total) {
  (void)total;
  if (MGR_IN(i, total, kDbgSmallOut)) p[i] = v;
}

// Plane `at` of `planes` in the shared memory of CTA `rank` (bounds-checking builds).
__device__ __forceinline__ bool slab_in(int rank, int at, int planes) {
  return MGR_IN(rank, kClusterSize, kDbgClusterRank) && MGR_IN(at, planes, kDbgClusterPlane);
}

// LOCAL: barrier of the CTA, else of the cluster.
template <bool LOCAL>
__device__ __forceinline__ void cluster_sync() {
  if (LOCAL) __syncthreads();
  else cooperative_groups::this_cluster().sync();
}

// Same address in CTA `rank`'s shared memory.
template <typename T>
__device__ __forceinline__ T* at_rank(T* p, int rank) {
  return cooperative_groups::this_cluster().map_shared_rank(p, rank);
}

// A = P_2 W on coarse planes q0 .. min(q1, m0 - 1) (the own and the next), m1 x n2
// values each; row(q, q1) gives the coarse values, `fine`: at the even places of the
// level's own rows (the last one at n2 - 1).
template <bool FINE, typename TS, typename TW, typename Row>
__device__ __forceinline__ void cluster_rows(const ClusterLevel<TS, TW>& g, TS* A, Row row) {
  const int planes = g.q0 < g.q1 ? min(g.q1 + 1, g.m0) - g.q0 : 0;
  const SmallDiv dn2(g.n2), dm1(g.m1);
  for (int e = threadIdx.x; e < planes * g.m1 * g.n2; e += kClusterThreads) {
    int i2, q1;
    const int q = dm1.quo_rem(dn2.quo_rem(e, i2), q1);
    const TW* r = row(g.q0 + q, q1);
    if (is_coarse(i2, g.n2)) A[e] = TS(r[FINE ? i2 : cidx(i2)]);
    else A[e] = g.wa[2][i2] * TS(r[FINE ? i2 - 1 : cidx(i2 - 1)]) + g.wb[2][i2] * TS(r[FINE ? i2 + 1 : cidx(i2 + 1)]);
  }
}
// The y and then z interpolation of A at level node (i0, i1, i2).
template <typename TS, typename TW>
__device__ __forceinline__ TS cluster_interp(const ClusterLevel<TS, TW>& g, const TS* A, int i0, int i1, int i2) {
  auto plane = [&](int q) -> TS {
    const TS* p = A + (q - g.q0) * g.m1 * g.n2 + i2;
    if (is_coarse(i1, g.n1)) return p[cidx(i1) * g.n2];
    return g.wa[1][i1] * p[cidx(i1 - 1) * g.n2] + g.wb[1][i1] * p[cidx(i1 + 1) * g.n2];
  };
  if (is_coarse(i0, g.n0)) return plane(cidx(i0));
  return g.wa[0][i0] * plane(cidx(i0 - 1)) + g.wb[0][i0] * plane(cidx(i0 + 1));
}

// Thomas solve of one line in place, U elements' loads ahead of the recurrence and
// their stores after it (U 16 with the last batch masked: 4100 cycles in FP64 for
// lines of 9, against 1700).
template <typename TW>
__device__ __forceinline__ void cluster_line(TW* f, int stride, int len, const TW* ta, const TW* tb) {
  constexpr int U = 4;
  TW prev = TW(0);
  int q = 0;
  for (; q + U <= len; q += U) {
    TW v[U], k[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      v[u] = f[(q + u) * stride];
      k[u] = ta[q + u];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      prev = v[u] - k[u] * prev;
      v[u] = prev;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) f[(q + u) * stride] = v[u];
  }
#pragma unroll 1
  for (; q < len; ++q) {
    prev = f[q * stride] - ta[q] * prev;
    f[q * stride] = prev;
  }
  TW next = TW(0);
  for (q = len - 1; q >= U - 1; q -= U) {
    TW v[U], k[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      v[u] = f[(q - u) * stride];
      k[u] = tb[q - u];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      next = v[u] - k[u] * next;
      v[u] = next;
    }
#pragma unroll
    for (int u = 0; u < U; ++u) f[(q - u) * stride] = v[u];
  }
#pragma unroll 1
  for (; q >= 0; --q) {
    next = f[q * stride] - tb[q] * next;
    f[q * stride] = next;
  }
}

// z = the correction of the level from the coefficients c of the own planes: on
// return the own z lines are in fz (m0 values each, at stride per; line k of this CTA is
// node rank * per + k of a coarse plane), and every CTA has passed the load vector.
// LOCAL: the whole level is this CTA's, z in f.
template <bool LOCAL, typename TS, typename TW>
__device__ __forceinline__ void cluster_correction(const ClusterLevel<TS, TW>& g, const int* active, const TW* c,
                                                   TW* f, TW* fz, TS* t1, TS* t2, int rank, int per) {
  const int own = g.i1 - g.i0, ownc = g.q1 - g.q0, n1 = g.n1, n2 = g.n2, m1 = g.m1, m2 = g.m2, mm = m1 * m2;
  const SmallDiv dm2(m2), dm1(m1), dmm(mm), dper(per);
  // row q of K on the values v at stride st
  auto row = [](const TS* k, int q, int len, const auto* v, int st) -> TS {
    const int p = pidx(q, len);
    TS acc = TS(0);
#pragma unroll
    for (int o = 0; o < 5; ++o) {
      const int j = p + o - 2;
      if (j >= 0 && j < len) acc += k[5 * q + o] * TS(v[j * st]);
    }
    return acc;
  };
  for (int e = threadIdx.x; e < own * n1 * m2; e += kClusterThreads) {
    int q;
    const int r = dm2.quo_rem(e, q);
    t1[e] = row(g.k[2], q, n2, c + r * n2, 1);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < own * mm; e += kClusterThreads) {
    int x, q;
    const int i0 = dm1.quo_rem(dm2.quo_rem(e, x), q);
    t2[e] = row(g.k[1], q, n1, t1 + i0 * n1 * m2 + x, m2);
  }
  cluster_sync<LOCAL>();
  const SmallDiv dm0(g.m0);
  for (int e = threadIdx.x; e < ownc * mm; e += kClusterThreads) {
    int yx;
    const int q = g.q0 + dmm.quo_rem(e, yx), p = pidx(q, g.n0);
    TS acc = TS(0);
#pragma unroll
    for (int o = 0; o < 5; ++o) {
      const int j = p + o - 2;
      if (j < 0 || j >= g.n0) continue;
      const TS* t;
      if (LOCAL || (j >= g.i0 && j < g.i1)) {
        t = t2 + (j - g.i0) * mm;
      } else {  // a neighbour's plane
        const int rr = slab_owner(j == g.n0 - 1 ? g.m0 - 1 : j >> 1, dm0);
        const int plane = j - pidx(slab_start(rr, g.m0), g.n0);
        if (!slab_in(rr, plane, 2 * slab_planes(g.m0))) continue;
        t = at_rank(t2, rr) + plane * mm;
      }
      acc += g.k[0][5 * q + o] * t[yx];
    }
    f[e] = TW(acc);
  }
  __syncthreads();
  if (active[2]) {
    for (int li = threadIdx.x; li < ownc * m1; li += kClusterThreads) cluster_line(f + li * m2, 1, m2, g.ta[2], g.tb[2]);
    __syncthreads();
  }
  if (active[1]) {
    for (int li = threadIdx.x; li < ownc * m2; li += kClusterThreads) {
      int x;
      const int q = dm2.quo_rem(li, x);
      cluster_line(f + q * mm + x, m2, m1, g.ta[1], g.tb[1]);
    }
    __syncthreads();
  }
  if (LOCAL) {
    if (active[0]) {
      for (int li = threadIdx.x; li < mm; li += kClusterThreads) cluster_line(f + li, mm, g.m0, g.ta[0], g.tb[0]);
      __syncthreads();
    }
    return;
  }
  for (int e = threadIdx.x; e < ownc * mm; e += kClusterThreads) {
    int yx, k;
    const int q = g.q0 + dmm.quo_rem(e, yx), rr = dper.quo_rem(yx, k);
    if (!slab_in(rr, q, g.m0)) continue;
    at_rank(fz, rr)[q * per + k] = f[e];
  }
  cluster_sync<false>();
  if (active[0]) {
    const int lines = min(per, mm - rank * per);
    for (int li = threadIdx.x; li < lines; li += kClusterThreads) cluster_line(fz + li, per, g.m0, g.ta[0], g.tb[0]);
    __syncthreads();
  }
}


// Decomposition of level l (its values in V): see the head of the file.
template <bool LOCAL, typename TD, typename TS, typename TW>
__device__ __forceinline__ void coarse_dec_level(const ClusterArgs<TS, TW>& a, unsigned char* smem, int l, int rank) {
  const ClusterLevel<TS, TW> g = cluster_level<LOCAL>(a, smem, l, rank);
  const int n1 = g.n1, n2 = g.n2, m1 = g.m1, m2 = g.m2, mm = m1 * m2, ownc = g.q1 - g.q0;
  const SmallDiv dn1(n1), dn2(n2), dm0(g.m0), dm1(m1), dm2(m2);
  TW* const V = reinterpret_cast<TW*>(smem + a.v[l]);
  TW* const W = reinterpret_cast<TW*>(smem + a.w[0]);
  TW* const f = reinterpret_cast<TW*>(smem + a.f);
  TW* const fz = reinterpret_cast<TW*>(smem + a.fz);
  TS* const t1 = reinterpret_cast<TS*>(smem + a.t1);
  TS* const t2 = reinterpret_cast<TS*>(smem + a.t2);
  TD* const out = static_cast<TD*>(a.out);
  auto coarse_at = [&](int e) {  // the level node of own coarse node e
    int y, x;
    const int q = dm1.quo_rem(dm2.quo_rem(e, x), y);
    return ((pidx(g.q0 + q, g.n0) - g.i0) * n1 + pidx(y, n1)) * n2 + pidx(x, n2);
  };
  for (int e = threadIdx.x; e < ownc * mm; e += kClusterThreads) W[e] = V[coarse_at(e)];
  // (the plane of q1 is the first of the next slab)
  const TW* next = !LOCAL && g.q1 < g.m0 ? at_rank(V, slab_owner(g.q1, dm0)) : V;
  cluster_rows<true>(g, t1, [&](int q, int y) -> const TW* {
    return LOCAL || q < g.q1 ? V + ((pidx(q, g.n0) - g.i0) * n1 + pidx(y, n1)) * n2 : next + pidx(y, n1) * n2;
  });
  // (waited for where the coarse values, which the neighbours read, are cleared)
  if (!LOCAL) cooperative_groups::this_cluster().barrier_arrive();
  __syncthreads();
  // coefficients (in place), written to their nodal positions
  for (int e = threadIdx.x; e < (g.i1 - g.i0) * n1 * n2; e += kClusterThreads) {
    int i1, i2;
    const int i0 = g.i0 + dn1.quo_rem(dn2.quo_rem(e, i2), i1);
    if (is_coarse(i0, g.n0) && is_coarse(i1, n1) && is_coarse(i2, n2)) continue;
    const TS c = TS(V[e]) - cluster_interp(g, t1, i0, i1, i2);
    if (!LOCAL || (e / 32) % kClusterSize == rank)
      cluster_st(out, cluster_full(a, a.s[l], i0, i1, i2), TD(c), a.total);
    V[e] = TW(c);
  }
  if (!LOCAL) cooperative_groups::this_cluster().barrier_wait();
  for (int e = threadIdx.x; e < ownc * mm; e += kClusterThreads) V[coarse_at(e)] = TW(0);
  __syncthreads();
  const int per = LOCAL ? mm : (mm + kClusterSize - 1) / kClusterSize;
  cluster_correction<LOCAL>(g, a.active[l], V, f, fz, t1, t2, rank, per);
  // the corrected coarse values (Eq. (1)) are the next level, or the coarsest grid
  if (LOCAL) {
    TW* const V1 = reinterpret_cast<TW*>(smem + a.v[l > 1 ? l - 1 : 1]);
    for (int e = threadIdx.x; e < ownc * mm; e += kClusterThreads) {
      const TW v = W[e] + f[e];
      if (l > 1) {
        V1[e] = v;
      } else if ((e / 32) % kClusterSize == rank) {
        int y, x;
        const int q = dm1.quo_rem(dm2.quo_rem(e, x), y);
        cluster_st(out, cluster_full(a, a.s0, q, y, x), TD(v), a.total);
      }
    }
    __syncthreads();
    return;
  }
  const int lines = min(per, mm - rank * per);
  if (lines > 0) {
    const SmallDiv dl(lines), dk0(l > 1 ? a.m[l - 1][0] : 1);
    for (int e = threadIdx.x; e < g.m0 * lines; e += kClusterThreads) {
      int k;
      const int q = dl.quo_rem(e, k), yx = rank * per + k;
      const int from = slab_owner(q, dm0), at = q - slab_start(from, g.m0);
      if (!slab_in(from, at, slab_planes(g.m0))) continue;
      const TW v = at_rank(W, from)[at * mm + yx] + fz[q * per + k];
      if (l == 1) {
        int x;
        const int y = dm2.quo_rem(yx, x);
        cluster_st(out, cluster_full(a, a.s0, q, y, x), TD(v), a.total);
        continue;
      }
      TW* const V1 = reinterpret_cast<TW*>(smem + a.v[l - 1]);
      if (l - 1 <= a.local) {
#pragma unroll
        for (int to = 0; to < kClusterSize; ++to) at_rank(V1, to)[q * mm + yx] = v;
      } else {
        const int to = slab_owner(q == g.m0 - 1 ? dk0.d - 1 : q >> 1, dk0);
        const int plane = q - pidx(slab_start(to, dk0.d), g.m0);
        if (slab_in(to, plane, 2 * slab_planes(dk0.d))) at_rank(V1, to)[plane * mm + yx] = v;
      }
    }
  }
  cluster_sync<false>();
}

// Recomposition of level l from its coefficients in V and the coarse values W.
template <bool LOCAL, typename TD, typename TS, typename TW>
__device__ __forceinline__ void coarse_rec_level(const ClusterArgs<TS, TW>& a, unsigned char* smem, int l, int rank) {
  const ClusterLevel<TS, TW> g = cluster_level<LOCAL>(a, smem, l, rank);
  const int n1 = g.n1, n2 = g.n2, m2 = g.m2, mm = g.m1 * m2;
  const SmallDiv dn1(n1), dn2(n2), dm0(g.m0);
  TW* const V = reinterpret_cast<TW*>(smem + a.v[l]);
  TW* const W = reinterpret_cast<TW*>(smem + a.w[l & 1]);
  TW* const W1 = reinterpret_cast<TW*>(smem + a.w[(l + 1) & 1]);
  TW* const f = reinterpret_cast<TW*>(smem + a.f);
  TW* const fz = reinterpret_cast<TW*>(smem + a.fz);
  TS* const t1 = reinterpret_cast<TS*>(smem + a.t1);
  TS* const t2 = reinterpret_cast<TS*>(smem + a.t2);
  const int per = LOCAL ? mm : (mm + kClusterSize - 1) / kClusterSize;
  cluster_correction<LOCAL>(g, a.active[l], V, f, fz, t1, t2, rank, per);
  if (LOCAL) {
    for (int e = threadIdx.x; e < g.m0 * mm; e += kClusterThreads) W[e] -= f[e];
  } else {
    const int lines = min(per, mm - rank * per);
    if (lines > 0) {
      const SmallDiv dl(lines);
      for (int e = threadIdx.x; e < g.m0 * lines; e += kClusterThreads) {
        int k;
        const int q = dl.quo_rem(e, k), yx = rank * per + k;
        const int from = slab_owner(q, dm0), at = q - slab_start(from, g.m0);
        if (slab_in(from, at, slab_planes(g.m0))) at_rank(W, from)[at * mm + yx] -= fz[q * per + k];
      }
    }
  }
  cluster_sync<LOCAL>();
  // level values: coefficients plus the interpolant of the coarse values
  const TW* next = !LOCAL && g.q1 < g.m0 ? at_rank(W, slab_owner(g.q1, dm0)) : W;
  cluster_rows<false>(g, t1, [&](int q, int y) -> const TW* {
    return LOCAL || q < g.q1 ? W + ((q - g.q0) * g.m1 + y) * m2 : next + y * m2;
  });
  __syncthreads();
  const bool last = l == a.levels;
  const bool up_local = l + 1 <= a.local;
  const SmallDiv up(last ? 1 : a.m[l + 1][0]);
  const int up0 = up_local ? 0 : slab_start(rank, up.d), up1 = up_local ? g.n0 : slab_start(rank + 1, up.d);
  for (int e = threadIdx.x; e < (g.i1 - g.i0) * n1 * n2; e += kClusterThreads) {
    int i1, i2;
    const int i0 = g.i0 + dn1.quo_rem(dn2.quo_rem(e, i2), i1), i12 = i1 * n2 + i2;
    const bool coarse = is_coarse(i0, g.n0) && is_coarse(i1, n1) && is_coarse(i2, n2);
    TW v;
    if (coarse) v = W[((cidx(i0) - g.q0) * g.m1 + cidx(i1)) * m2 + cidx(i2)];
    else v = TW(TS(V[e]) + cluster_interp(g, t1, i0, i1, i2));
    if (!last) {  // a coarse plane of the next level
      if (LOCAL) {
        if (i0 >= up0 && i0 < up1) W1[(i0 - up0) * n1 * n2 + i12] = v;
      } else {
        const int to = slab_owner(i0, up), at = i0 - slab_start(to, up.d);
        if (slab_in(to, at, slab_planes(up.d))) at_rank(W1, to)[at * n1 * n2 + i12] = v;
      }
    } else if (!LOCAL || (e / 32) % kClusterSize == rank) {
      if (a.vout_full) cluster_st(static_cast<TD*>(a.vout), cluster_full(a, a.s[l], i0, i1, i2), TD(v), a.total);
      else cluster_st(static_cast<TW*>(a.vout), i0 * n1 * n2 + i12, v, g.n0 * n1 * n2);
    }
  }
  __syncthreads();
}

// The arguments, in shared memory: read from the constant cache a word at a time, cold,
// they took a quarter of the kernel's time.
template <typename TS, typename TW>
__device__ __forceinline__ void cluster_copy_args(const ClusterArgs<TS, TW>& from, ClusterArgs<TS, TW>& to) {
  static_assert(sizeof(from) % 8 == 0, "copied in words of 8 bytes");
  const unsigned long long* s = reinterpret_cast<const unsigned long long*>(&from);
  unsigned long long* d = reinterpret_cast<unsigned long long*>(&to);
  for (int i = threadIdx.x; i < int(sizeof(from) / 8); i += kClusterThreads) d[i] = s[i];
  __syncthreads();
}

template <typename TD, typename TS, typename TW>
__global__ void __cluster_dims__(kClusterSize, 1, 1) __launch_bounds__(kClusterThreads, 1)
    k_coarse_dec(const __grid_constant__ ClusterArgs<TS, TW> args) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) unsigned char args_raw[sizeof(ClusterArgs<TS, TW>)];
  ClusterArgs<TS, TW>& a = *reinterpret_cast<ClusterArgs<TS, TW>*>(args_raw);
  cluster_copy_args(args, a);
  auto cluster = cooperative_groups::this_cluster();
  const int rank = int(cluster.block_rank()), ls = a.levels;
  cluster_copy_tables(a, smem_raw);
  {
    const bool local = ls <= a.local;
    const ClusterLevel<TS, TW> g = local ? cluster_level<true>(a, smem_raw, ls, rank) : cluster_level<false>(a, smem_raw, ls, rank);
    const SmallDiv dn1(g.n1), dn2(g.n2);
    TW* V = reinterpret_cast<TW*>(smem_raw + a.v[ls]);
    const int first = g.i0 * g.n1 * g.n2;
#pragma unroll 4
    for (int e = threadIdx.x; e < (g.i1 - g.i0) * g.n1 * g.n2; e += kClusterThreads) {
      if (a.vin_full) {
        int i1, i2;
        const int i0 = g.i0 + dn1.quo_rem(dn2.quo_rem(e, i2), i1);
        V[e] = TW(cluster_ld(static_cast<const TD*>(a.vin), cluster_full(a, a.s[ls], i0, i1, i2), a.total));
      } else {
        V[e] = cluster_ld(static_cast<const TW*>(a.vin), first + e, g.n0 * g.n1 * g.n2);
      }
    }
  }
  cp_wait<0>();
  cluster.sync();  // (the output may be the input)
  int l = ls;
  for (; l > a.local; --l) coarse_dec_level<false, TD>(a, smem_raw, l, rank);
  for (; l >= 1; --l) coarse_dec_level<true, TD>(a, smem_raw, l, rank);
}

template <typename TD, typename TS, typename TW>
__global__ void __cluster_dims__(kClusterSize, 1, 1) __launch_bounds__(kClusterThreads, 1)
    k_coarse_rec(const __grid_constant__ ClusterArgs<TS, TW> args) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) unsigned char args_raw[sizeof(ClusterArgs<TS, TW>)];
  ClusterArgs<TS, TW>& a = *reinterpret_cast<ClusterArgs<TS, TW>*>(args_raw);
  cluster_copy_args(args, a);
  auto cluster = cooperative_groups::this_cluster();
  const int rank = int(cluster.block_rank()), ls = a.levels;
  cluster_copy_tables(a, smem_raw);
  const TD* cin = static_cast<const TD*>(a.cin);
  // the coarsest values, and the coefficients of every level's own planes (0 on
  // coarse nodes)
  for (int l = ls; l >= 1; --l) {
    const ClusterLevel<TS, TW> g = l <= a.local ? cluster_level<true>(a, smem_raw, l, rank) : cluster_level<false>(a, smem_raw, l, rank);
    const SmallDiv dn1(g.n1), dn2(g.n2), dm1(g.m1), dm2(g.m2);
    if (l == 1)
      for (int e = threadIdx.x; e < (g.q1 - g.q0) * g.m1 * g.m2; e += kClusterThreads) {
        int y, x;
        const int q = g.q0 + dm1.quo_rem(dm2.quo_rem(e, x), y);
        reinterpret_cast<TW*>(smem_raw + a.w[1])[e] = TW(cluster_ld(cin, cluster_full(a, a.s0, q, y, x), a.total));
      }
    TW* V = reinterpret_cast<TW*>(smem_raw + a.v[l]);
#pragma unroll 4
    for (int e = threadIdx.x; e < (g.i1 - g.i0) * g.n1 * g.n2; e += kClusterThreads) {
      int i1, i2;
      const int i0 = g.i0 + dn1.quo_rem(dn2.quo_rem(e, i2), i1);
      const bool coarse = is_coarse(i0, g.n0) && is_coarse(i1, g.n1) && is_coarse(i2, g.n2);
      V[e] = coarse ? TW(0) : TW(cluster_ld(cin, cluster_full(a, a.s[l], i0, i1, i2), a.total));
    }
  }
  cp_wait<0>();
  // (the output may be the input; every CTA has started before its memory is read)
  cluster.sync();
  int l = 1;
  for (; l <= a.local; ++l) coarse_rec_level<true, TD>(a, smem_raw, l, rank);
  for (; l <= ls; ++l) coarse_rec_level<false, TD>(a, smem_raw, l, rank);
  cluster.sync();  // a CTA's shared memory is read until here
}
