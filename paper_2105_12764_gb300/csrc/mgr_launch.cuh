// mgr_launch.cuh -- host-side launch helpers shared by the level loops of
// the single-field paths (mgr_core.cu: 1D-3D; mgr_st.cu: the spatiotemporal
// 4D form): per-launch event recording, plan tables, level arguments, grid
// choices, kernel launches of the level pass / interpolation / solves and the
// coarsest-grid copy.  Included inside an anonymous namespace after the kernel
// headers (mgr_device.cuh, mgr_level.cuh, mgr_solve.cuh).
#pragma once

// Optional per-launch CUDA-event instrumentation (mgr_profile).
inline void rec_begin(cudaStream_t st) {
  if (!t_recorder) return;
  LaunchRecord r{};
  cudaEventCreate(&r.start);
  cudaEventCreate(&r.stop);
  cudaEventRecord(r.start, st);
  t_recorder->launches.push_back(r);
}
inline void rec_end(cudaStream_t st, const char* name, int level, double bytes, double flops) {
  if (!t_recorder) return;
  LaunchRecord& r = t_recorder->launches.back();
  cudaEventRecord(r.stop, st);
  std::snprintf(r.name, sizeof(r.name), "%s", name);
  r.level = level;
  r.bytes = bytes;
  r.flops = flops;
}

// ---------------------------------------------------------------------------
// Host-side level loops
// ---------------------------------------------------------------------------

template <typename T>
const T* table(const mgr_plan* p);
template <>
const double* table<double>(const mgr_plan* p) { return p->tables.d64; }
template <>
const float* table<float>(const mgr_plan* p) { return p->tables.d32; }

inline int grid_1d(int64_t total, int block, const mgr_plan* p) {
  int64_t g = (total + block - 1) / block;
  int64_t cap = int64_t(p->ctx->num_sms) * 32;
  return int(std::max<int64_t>(1, std::min(g, cap)));
}

struct Bufs {
  void* A;
  void* B;
  void* F;
};

inline Bufs split_ws(const mgr_plan* p, void* ws) {
  char* b = static_cast<char*>(ws);
  return Bufs{b, b + p->ws_a, b + p->ws_a + p->ws_b};
}

template <typename TS, typename TW>
LevelArgs<TS, TW> level_args(const mgr_plan* p, int l) {
  const LevelGeom& g = p->geom[l];
  LevelArgs<TS, TW> a{};
  const TS* T = table<TS>(p);
  for (int k = 0; k < 3; ++k) {
    a.n[k] = g.ax[k].n;
    a.m[k] = g.ax[k].m;
    a.s[k] = g.ax[k].s;
    a.N[k] = g.ax[k].N;
    a.slot[k] = T + g.ax[k].o_slot;
  }
  a.y_sz = p->full[1] * p->full[2];
  a.y_sy = p->full[2];
  a.c_sz = int64_t(g.ax[1].m) * g.ax[2].m;
  a.c_sy = g.ax[2].m;
  return a;
}

// Strip height and z chunk length of the warp-per-strip passes (level pass,
// interpolation) over my x mz coarse rows and planes.  A warp streams rows +
// `row_halo` units per plane pair over its chunk's planes and `plane_halo` more:
// long strips and chunks repeat least, short ones make more warps.  The model:
// with c warps on an SM a unit takes max(rate, chain / c) cycles of it, `rate` what
// bounds the pass and `chain` one warp's own latency.  Up to two rounds of resident
// warps are counted as such, the last one with the warps it has; of more rounds
// than that, whose warps end one by one, half a warp's time is lost at the end.
// tile > 0: only heights that divide it.
struct StripShape {
  int rows = 1, chunk = 1;
};
struct StripModel {
  double rate, chain, row_halo, plane_halo;
  int max_rows, tile;
};
template <typename Warps, typename Resident>
StripShape strip_shape(const mgr_plan* p, int my, int mz, const StripModel& md, Warps warps_of, Resident resident_of) {
  const int64_t sms = p->ctx->num_sms;
  StripShape out;
  double best = 1e300;
  for (int rows = 1; rows <= md.max_rows; ++rows) {
    if (md.tile > 0 && md.tile % rows != 0) continue;
    const int strips = (my + rows - 1) / rows;
    const int r = md.tile > 0 ? rows : (my + strips - 1) / strips;  // evenly over the strips
    const int64_t warps = warps_of(r), resident = resident_of(r);
    // every chunk length that splits the planes evenly, longest first
    for (int len = mz;;) {
      const int chunks = (mz + len - 1) / len;
      const int even = (mz + chunks - 1) / chunks;
      const int64_t w = warps * chunks;
      const double units = (r + md.row_halo) * (even + (mz > 1 ? md.plane_halo : 0.0));
      const int64_t full = w / (sms * resident), rest = (w - full * sms * resident + sms - 1) / sms;
      const double round = std::max(md.rate * resident, md.chain);
      const double cost =
          units * (full < 2 ? full * round + (rest > 0 ? std::max(md.rate * rest, md.chain) : 0.0)
                            : (double(w) / sms + 0.5) * round / resident);
      if (cost < best * (1 - 1e-9)) {
        best = cost;
        out = StripShape{r, even};
      }
      if (even <= 1) break;
      len = even - 1;
    }
    if (rows >= my) break;
  }
  return out;
}
inline int64_t resident_warps(size_t smem, int limit) {
  return std::min<int64_t>(limit, (int64_t(227) << 10) / int64_t(smem + 1024));
}

// Shape of the level pass (sets a.rows, a.qz_chunk) for `slices` grids of the level
// at once, `planes` coarse planes of each.  Rates: FP64 49 / 32 operations of 16
// cycles; FP32 the instructions and the shared-memory and shuffle pipe, measured
// at 513^3.  Chains: measured with few warps.  FP32 strips have at most 10 rows:
// longer ones take the L1 cache's share of the memory (513^3: 0.29 ms with 8 or
// 10 rows, 0.33 with 12 to 14).  FP32 codes have strips of 7, 2 or 1 rows, which
// lie in one of the runs of 14 whose places decide a rounding (see level_body).
template <int MODE, typename TI, bool QZ, typename TS, typename TW>
void level_shape(const mgr_plan* p, LevelArgs<TS, TW>& a, int64_t slices = 1, int planes = 1 << 30) {
  constexpr bool F64 = sizeof(TS) == 8;
  constexpr bool codes = QZ && MODE == 0 && !F64;
  const StripModel md{F64 ? (MODE == 0 ? 784.0 : 512.0) : (MODE == 0 ? 110.0 : 62.0),
                      F64 ? (MODE == 0 ? 4200.0 : 2900.0) : (MODE == 0 ? 1000.0 : 620.0),
                      1.5,
                      1.2,
                      F64 ? 16 : codes ? 7 : 10,
                      codes ? 14 : 0};
  const int my = a.m[1], mx = a.m[2];
  const StripShape s = strip_shape(
      p, my, std::min(a.m[0], planes), md, [&](int r) { return level_warps<32>(mx, my, r) * slices; },
      [&](int r) {
        return resident_warps(level_smem_bytes<MODE, TI, TS, QZ>(r, level_slot_rows(mx, my, r)), level_ctas<MODE, TS>());
      });
  a.rows = s.rows;
  a.qz_chunk = s.chunk;
}

// Grid of the level pass: warps over the strips, z chunks (sets a.rows, a.qz_chunk;
// chosen for `planes` coarse planes at a time).
template <int MODE, typename TI, bool QZ, typename TS, typename TW>
dim3 level_grid(const mgr_plan* p, LevelArgs<TS, TW>& a, int planes = 1 << 30) {
  level_shape<MODE, TI, QZ>(p, a, 1, planes);
  return dim3(unsigned(level_warps<32>(a.m[2], a.m[1], a.rows)), (a.m[0] + a.qz_chunk - 1) / a.qz_chunk);
}

// spread: a grid of one round asks for as much shared memory as lets every SM
// hold its even share of the warps and no more.  Beside other kernels the
// warps would otherwise pile up, to twice the share, on the SMs that happen to
// be free when the pass starts: FP64 recomposition of 385^3 1.38 to 1.83 ms
// without, 1.14 with; 321^3 0.92, 0.75.
//
// z chunks [c0, c1) of the level pass's grid (the grid level_grid chooses with
// `planes`; c1 < 0: all of them): a level pass may run as several such launches,
// each as soon as its input planes are ready.
template <int MODE, typename TI, typename TD, typename TS, typename TW, bool PK, bool QZ = false>
void launch_level_chunks(const mgr_plan* p, LevelArgs<TS, TW>& a, int c0, int c1, cudaStream_t st,
                         int planes = 1 << 30, bool spread = false) {
  dim3 grid = level_grid<MODE, TI, QZ>(p, a, planes);
  if (c1 < 0) c1 = int(grid.y);
  if (c1 <= c0 || c1 > int(grid.y)) return;
  size_t sm = level_smem_bytes<MODE, TI, TS, QZ>(a.rows, level_slot_rows(a.m[2], a.m[1], a.rows));
  if (spread) {
    const int64_t each = (int64_t(grid.x) * (c1 - c0) + p->ctx->num_sms - 1) / p->ctx->num_sms;
    if (each <= resident_warps(sm, level_ctas<MODE, TS>()))
      sm = std::max(sm, ((size_t(227) << 10) / size_t(each) - 1024) / 128 * 128);
  }
  auto kern = k_level<MODE, TI, TD, TS, TW, true, PK, QZ>;
  if constexpr (!PK) {
    if (a.s[2] != 1) kern = k_level<MODE, TI, TD, TS, TW, false, PK, QZ>;
  }
  raise_smem_limit(kern, sm);
  // (the grid's y extent is limited to 65535)
  for (int c = c0; c < c1; c += 65535) {
    a.bz0 = c;
    grid.y = unsigned(std::min(c1 - c, 65535));
    kern<<<grid, 32, sm, st>>>(a);
  }
  a.bz0 = 0;
}

template <int MODE, typename TI, typename TD, typename TS, typename TW, bool PK, bool QZ = false>
void launch_level(const mgr_plan* p, LevelArgs<TS, TW>& a, cudaStream_t st, bool spread = false) {
  launch_level_chunks<MODE, TI, TD, TS, TW, PK, QZ>(p, a, 0, -1, st, 1 << 30, spread);
}

// c: nodal coefficients (PK false), the packed class of level l (PK true), or
// null for a dropped class (all coefficients zero); QZ: c holds codes of bin
// width qs
template <typename TD, typename TO, typename TS, typename TW, bool PK, bool QZ = false>
void launch_interp(const mgr_plan* p, int l, const void* c, const TW* w, void* out, int out_full, cudaStream_t st,
                   double qs = 1.0);

// Arguments of the interpolation of level l (spatial axes); its shape is left to
// the caller.
template <typename TS, typename TW, bool PK = false>
InterpArgs<TS, TW> interp_args(const mgr_plan* p, int l, const void* c, const TW* w, void* out, int out_full,
                               double qs) {
  const LevelGeom& g = p->geom[l];
  const TS* T = table<TS>(p);
  InterpArgs<TS, TW> a{};
  for (int k = 0; k < 3; ++k) {
    a.n[k] = g.ax[k].n;
    a.m[k] = g.ax[k].m;
    a.s[k] = g.ax[k].s;
    a.N[k] = g.ax[k].N;
    a.slot[k] = T + g.ax[k].o_slot;
  }
  a.c = c;
  a.y_sz = PK ? int64_t(g.ax[1].n) * g.ax[2].n : p->full[1] * p->full[2];
  a.y_sy = PK ? int64_t(g.ax[2].n) : p->full[2];
  a.w = w;
  a.c_sz = int64_t(g.ax[1].m) * g.ax[2].m;
  a.c_sy = g.ax[2].m;
  a.out = out;
  a.qs = qs;
  a.o_sz = out_full ? p->full[1] * p->full[2] : int64_t(g.ax[1].n) * g.ax[2].n;
  a.o_sy = out_full ? p->full[2] : int64_t(g.ax[2].n);
  return a;
}

// Shape of an interpolation (sets a.rows, a.qz_chunk) for `slices` grids of the
// level at once, `planes` coarse planes of each.  Rates: FP64 17 operations of 16
// cycles; FP32 a unit's 2.2 KB at an SM's share of the HBM.  Strips are short (FP32
// at most 4 rows, FP64 8): their interpolants take little shared memory, and the
// L1 cache, through which both columns of a row and the coarse values of
// neighbouring strips come, keeps the rest (513^3 FP32: 0.22 ms with 4 rows, 0.23
// with 6, 0.27 with 8; FP64 0.59 with 4 or 8, 0.65 with 10 to 16).
template <typename TD, typename TS, typename TW>
void interp_shape(const mgr_plan* p, InterpArgs<TS, TW>& a, int64_t slices = 1, int planes = 1 << 30) {
  constexpr bool F64 = sizeof(TS) == 8;
  const StripModel md{F64 ? 270.0 : 102.0, F64 ? 3300.0 : 1050.0, 0.5, 0.4, F64 ? 8 : 4, 0};
  const int my = a.m[1], mx = a.m[2];
  const StripShape s = strip_shape(
      p, my, std::min(a.m[0], planes), md, [&](int r) { return interp_warps(mx, my, r) * slices; },
      [&](int r) { return resident_warps(interp_smem_bytes<TD, TS, TW>(r, level_slot_rows(mx, my, r)), 16); });
  a.rows = s.rows;
  a.qz_chunk = s.chunk;
}

// z chunks [c0, c1) of the interpolation of level l, its shape chosen for `planes`
// coarse planes at a time (c1 < 0: all of them)
template <typename TD, typename TO, typename TS, typename TW, bool PK, bool QZ>
void launch_interp_chunks(const mgr_plan* p, int l, const void* c, const TW* w, void* out, int out_full,
                          cudaStream_t st, double qs, int c0, int c1, int planes = 1 << 30) {
  InterpArgs<TS, TW> a = interp_args<TS, TW, PK>(p, l, c, w, out, out_full, qs);
  interp_shape<TD>(p, a, 1, planes);
  const int gz = (a.m[0] + a.qz_chunk - 1) / a.qz_chunk;
  if (c1 < 0) c1 = gz;
  if (c1 <= c0 || c1 > gz) return;
  const size_t sm = interp_smem_bytes<TD, TS, TW>(a.rows, level_slot_rows(a.m[2], a.m[1], a.rows));
  auto kern = k_interp<TD, TO, TS, TW, true, PK, QZ>;
  if constexpr (!PK) {
    if (a.s[2] != 1) kern = k_interp<TD, TO, TS, TW, false, PK, QZ>;
  }
  raise_smem_limit(kern, sm);
  // (the grid's y extent is limited to 65535)
  for (int k = c0; k < c1; k += 65535) {
    a.bz0 = k;
    kern<<<dim3(unsigned(interp_warps(a.m[2], a.m[1], a.rows)), unsigned(std::min(c1 - k, 65535))), 32, sm, st>>>(a);
  }
}

template <typename TD, typename TO, typename TS, typename TW, bool PK, bool QZ>
void launch_interp(const mgr_plan* p, int l, const void* c, const TW* w, void* out, int out_full, cudaStream_t st,
                   double qs) {
  launch_interp_chunks<TD, TO, TS, TW, PK, QZ>(p, l, c, w, out, out_full, st, qs, 0, -1);
}

// Thomas solves along the contiguous axis: `lines` lines of length mx,
// consecutive in memory.  Build-time knobs: MGR_X_SOLVE_ROWS (1: FP64 with
// many lines through k_solve_rows), MGR_X_SOLVE_KB (shared memory per CTA of
// k_solve_contig).
#ifndef MGR_X_SOLVE_ROWS
#define MGR_X_SOLVE_ROWS 1
#endif
#ifndef MGR_X_SOLVE_KB
#define MGR_X_SOLVE_KB 32
#endif
template <typename TW>
cudaError_t launch_x_solve(const mgr_plan* p, TW* f, TW* w, int mx, int64_t lines, const TW* ta, const TW* tb, int op,
                           cudaStream_t st) {
  (void)p;
  if (MGR_X_SOLVE_ROWS && sizeof(TW) == 8 && lines >= 32768) {
    // lines through 32 x 32 tiles, the intermediate through memory
    const int64_t nwarps = (lines + 31) / 32;
    k_solve_rows<TW><<<int((nwarps + kRowsWarps - 1) / kRowsWarps), kRowsWarps * 32, 0, st>>>(f, w, mx, lines, mx, ta,
                                                                                             tb, op);
    return cudaGetLastError();
  }
  if (solve_contig_smem<TW>(mx, 1) > 96 * 1024) {
    // lines too long to stage in shared memory: one thread per line from global memory
    const int blocks = int((lines + kStridedThreads - 1) / kStridedThreads);
    k_solve_strided<TW><<<blocks, kStridedThreads, 0, st>>>(f, w, mx, 1, 1, lines, mx, ta, tb, op);
    return cudaGetLastError();
  }
  const int pitch = contig_pitch<TW>(mx);
  // rows per CTA (one solving thread per row, 128 threads load and store): up
  // to 32, a whole warp of recurrences, within MGR_X_SOLVE_KB of shared memory
  int R = int(std::min<size_t>(32, (size_t(MGR_X_SOLVE_KB) * 1024) / (sizeof(TW) * pitch)));
  R = std::max(1, R);
  const size_t sm = solve_contig_smem<TW>(mx, R);
  const int blocks = int((lines + R - 1) / R);
  raise_smem_limit(k_solve_contig<TW>, sm);
  k_solve_contig<TW><<<blocks, 128, sm, st>>>(f, w, mx, lines, R, ta, tb, op);
  return cudaGetLastError();
}

template <typename TW>
cudaError_t solve_axis_launch(const mgr_plan* p, int l, int axis, TW* f, TW* w, int op, cudaStream_t st);

template <typename TW>
cudaError_t solve_axis(const mgr_plan* p, int l, int axis, TW* f, TW* w, int op, cudaStream_t st) {
  const Work wk = work_solve(p, l, axis, op != SOLVE_INPLACE);
  static const char* names[3] = {"solve_z", "solve_y", "solve_x"};
  rec_begin(st);
  cudaError_t err = solve_axis_launch<TW>(p, l, axis, f, w, op, st);
  rec_end(st, names[axis], l, wk.bytes, wk.flops);
  return err;
}

// Strided axes: whole lines staged in shared memory below this many lines
// (build-time knobs), one thread per line from global memory above.
#ifndef MGR_STAGED_LINES_F32
#define MGR_STAGED_LINES_F32 32768
#endif
#ifndef MGR_STAGED_LINES_F64
#define MGR_STAGED_LINES_F64 32768
#endif
template <typename TW>
cudaError_t solve_axis_launch(const mgr_plan* p, int l, int axis, TW* f, TW* w, int op, cudaStream_t st) {
  const LevelGeom& g = p->geom[l];
  const int mz = g.ax[0].m, my = g.ax[1].m, mx = g.ax[2].m;
  const TW* T = table<TW>(p);
  const TW* ta = T + g.ax[axis].o_ta;
  const TW* tb = T + g.ax[axis].o_tb;
  const int64_t lines_x = int64_t(mz) * my;
  if (axis == 2) return launch_x_solve<TW>(p, f, w, mx, lines_x, ta, tb, op, st);
  int mline, inner;
  int64_t lstride, outer, ostride;
  if (axis == 1) {
    mline = my; lstride = mx; inner = mx; outer = mz; ostride = int64_t(my) * mx;
  } else {
    mline = mz; lstride = int64_t(my) * mx; inner = mx; outer = my; ostride = mx;
  }
  const int64_t lines = int64_t(inner) * outer;
  const int64_t staged_below = sizeof(TW) == 4 ? int64_t(MGR_STAGED_LINES_F32) : int64_t(MGR_STAGED_LINES_F64);
  if (lines < staged_below) {
    // few lines (coarse levels, planes): whole lines staged in shared memory, fewer
    // per CTA where there would not be two CTAs per SM, or where they would not fit
    const int64_t want = 2 * int64_t(p->ctx->num_sms);
    const size_t limit = std::min<size_t>(size_t(220) * 1024, p->ctx->smem_optin);
    for (int nl : {32, 16, 8}) {
      const size_t ssm = solve_staged_smem<TW>(mline, nl);
      if (ssm > limit || (nl > 8 && lines < want * nl)) continue;
      auto kern = nl == 32 ? k_solve_staged<TW, 32> : nl == 16 ? k_solve_staged<TW, 16> : k_solve_staged<TW, 8>;
      raise_smem_limit(kern, ssm);
      kern<<<unsigned((lines + nl - 1) / nl), kStagedThreads, ssm, st>>>(f, w, mline, lstride, inner, outer, ostride,
                                                                           ta, tb, op);
      return cudaGetLastError();
    }
  }
  const int blocks = int((lines + kStridedThreads - 1) / kStridedThreads);
  k_solve_strided<TW><<<blocks, kStridedThreads, 0, st>>>(f, w, mline, lstride, inner, outer, ostride, ta, tb, op);
  return cudaGetLastError();
}

// solve along every active axis, x first; the last one applies `final_op` into w
template <typename TW>
cudaError_t solve_level(const mgr_plan* p, int l, TW* f, TW* w, int final_op, cudaStream_t st) {
  const LevelGeom& g = p->geom[l];
  int last = -1;
  for (int axis = 2; axis >= 0; --axis)
    if (g.ax[axis].active) last = axis;
  for (int axis = 2; axis >= 0; --axis) {
    if (!g.ax[axis].active) continue;
    cudaError_t e = solve_axis<TW>(p, l, axis, f, w, axis == last ? final_op : SOLVE_INPLACE, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// Coarsest grid <-> its place in the output: the nodal positions at stride
// 2^L (nodal layout) or class 0, the compact coarsest grid (packed layout).
template <typename TD, typename TW>
cudaError_t coarsest_copy_launch(const mgr_plan* p, TD* y, TW* w, bool packed, int dir, cudaStream_t st) {
  const int L = p->levels;
  const int3 n0 = make_int3(int(p->coarsest[0]), int(p->coarsest[1]), int(p->coarsest[2]));
  const int64_t s0 = packed ? 1 : (int64_t(1) << L);
  const longlong3 s = make_longlong3(p->full[0] > 1 ? s0 : 1, p->full[1] > 1 ? s0 : 1, s0);
  const longlong3 N = packed ? make_longlong3(n0.x, n0.y, n0.z) : make_longlong3(p->full[0], p->full[1], p->full[2]);
  const int64_t total = int64_t(n0.x) * n0.y * n0.z;
  rec_begin(st);
  k_coarsest<TD, TW><<<grid_1d(total, 256, p), 256, 0, st>>>(y, N.y * N.z, N.z, w, n0, s, N, dir);
  cudaError_t e = cudaGetLastError();
  rec_end(st, "coarsest", 0, double(total) * (sizeof(TD) + sizeof(TW)), 0.0);
  return e;
}
