// mgr_level.cuh -- the level pass of decomposition (coefficients + load
// vector) and the load-vector pass of recomposition, for sm_103a.
//
// Per level l (level grid n -> coarse grid m), one warp owns a strip of coarse
// y rows and a chunk of coarse z planes for the coarse x nodes of its lanes.
// It streams the fine z planes of its region in pairs -- the coarse-in-z plane
// p(t) and the fine-in-z plane between p(t-1) and p(t) -- and each plane pair in
// units of row pairs: the coarse row p(qc) and the fine row above it.  No step
// needs another warp, so there is no CTA barrier and no shared tile; a CTA is
// one warp, and its plane and row bookkeeping is the same for all lanes.
//
// Lanes.  Lane l owns one coarse x node and the fine node after it (two level
// columns).  The nodes of all strips of the level, one strip after another,
// form one sequence; a row group of LX lanes (a warp, or half of one) takes LX
// consecutive entries and shares two of them with its neighbours, so that each
// lane with outputs has its left and right neighbour in the group (warp
// shuffles) whatever the level's width: 30 of 32 lanes produce outputs on every
// grid, where tiles 30 nodes wide left almost half of them idle at 33.  Where a
// strip ends inside a group, the neighbour from the other strip carries weight 0.
//
// Coefficients (Sec. II.A.1), separable and in the paper's FMA form (Table
// "fma"): the x interpolant of a coarse row uses the right neighbour's value; the
// y interpolant of the fine row above lies between this coarse row's interpolants
// and the previous one's (kept from the previous unit); a fine-z plane
// interpolates between the xy interpolants of its two coarse planes, the first
// plane's kept in the lane's own shared-memory slots, one per unit.
//
// Load vector f' = (x_k D_k^-1 K_k) c (Sec. II.A.2, III.A.2): the x stencil of
// each row takes the neighbours' columns by shuffles (two taps on the rows coarse
// in y and z, where c vanishes on coarse nodes); the y stencil of coarse row qc-1
// is complete once unit qc's rows are there, from results kept in registers; the
// z stencil accumulates over the planes in the lane's shared-memory slots.
//
// Loads.  Asynchronous 4- or 8-byte copies into a ring of units in shared memory,
// three units ahead in FP32 (one in FP64): with the next unit's loads in
// registers the FP32 pass waited for them (0.83 ms at 513^3, against 0.30).
//
// What bounds it.  FP64: the FP64 pipe, one SM-wide operation per 16 cycles and
// warp; a unit takes 49 of them in decomposition, 32 in recomposition (level_shape
// counts with that); busy 91% of the finest pass at 257^3.  FP32: no single unit
// (385^3, finest level: issue slots 43%, shared-memory and shuffle pipe 67%, DRAM
// 52%), but the dependent chains of about 11 warps per
// SM.  513^3, finest level, against the earlier pass of 8-warp tiles with two CTA
// barriers per plane pair: FP64 decomposition 2.12 -> 1.82 ms, recomposition 1.48
// -> 1.12 ms; FP32 0.375 -> 0.303 and 0.248 -> 0.174 ms.  65^3 FP64, where the
// tiles left most SMs without work: 49 -> 24 us.
//
// Coefficient addressing.  Nodal (PK = false): a coefficient sits at its node's
// full-grid position.  Class-packed (PK = true, Sec. I coefficient classes): the
// coefficients of level l form one contiguous class, in row-major order of the
// level grid with the nodes of the coarser grid left out.  With cb(i) = (i+1)/2
// coarse nodes before index i, node (i, j, k) of class l is at
//   i*n1*n2 - cb(i)*m1*m2 + (i fine ? j*n2 + k
//                                   : j*n2 - cb(j)*m2 + (j fine ? k : k - cb(k)))
// from the class start, so plane and row offsets stay separable.
//
// Quantized coefficients (QZ, class-packed only): decomposition writes the
// int32 code round_half_even(c * (1/q_l)) of each coefficient (the rounding
// decision in the stencil type TS) and recomposition reads codes and uses
// code * q_l; q_l is the bin width of the level's class.
#pragma once

template <typename T>
struct Pair;
template <>
struct Pair<float> {
  using type = float2;
};
template <>
struct Pair<double> {
  using type = double2;
};
template <>
struct Pair<int> {
  using type = int2;
};

// int32 code of value v for 1/bin width qinv: v * qinv rounded to FP32 / FP64
// (no contraction), then rounded half to even; values whose code does not fit
// in (-2^31, 2^31) (and NaN) become +-(2^31-1) and are counted.
__device__ __forceinline__ int quant_code(float v, float qinv, unsigned long long* sat) {
  const float t = __fmul_rn(v, qinv);
  const float r = rintf(t);
  if (!(fabsf(r) < 2147483648.0f)) {
    if (sat) atomicAdd(sat, 1ull);
    return t > 0.0f ? 2147483647 : -2147483647;
  }
  return int(r);
}
// FP64: the product is the only FP64 operation; t is rounded to an integer
// from its IEEE-754 fields with integer instructions (the FP64 pipe, which
// bounds the FP64 level pass, has a small fraction of the integer pipes'
// throughput).  With t = 1.m * 2^e and the 53-bit significand M = 1m,
// |t| < 0.5 for e < -1; otherwise floor|t| = M >> (52 - e) and the
// remainder decides round-half-to-even.
__device__ __forceinline__ int quant_code(double v, double qinv, unsigned long long* sat) {
  const double t = __dmul_rn(v, qinv);
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(t));
  const int e = int((b >> 52) & 0x7ffu) - 1023;
  if (e < -1) return 0;
  const bool neg = (b >> 63) != 0;
  if (e <= 30) {
    const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
    const int sh = 52 - e;  // 22 .. 53
    unsigned long long q = m >> sh;
    const unsigned long long rem = m & ((1ull << sh) - 1), half = 1ull << (sh - 1);
    if (rem > half || (rem == half && (q & 1ull))) ++q;
    if (q < (1ull << 31)) return neg ? -int(q) : int(q);
  }
  if (sat) atomicAdd(sat, 1ull);
  const bool nan = e == 1024 && (b & 0xFFFFFFFFFFFFFull) != 0;
  return (!neg && !nan) ? 2147483647 : -2147483647;
}

// Code k as a value of the stencil type.  FP64 assembles the IEEE-754 fields
// of the (exactly representable) integer with integer instructions: sign,
// exponent 1023 + msb(|k|), and |k| shifted up to the 52-bit fraction.
template <typename TS>
__device__ __forceinline__ TS code_value(int k);
template <>
__device__ __forceinline__ float code_value<float>(int k) {
  return float(k);
}
template <>
__device__ __forceinline__ double code_value<double>(int k) {
  const unsigned s = unsigned(k) & 0x80000000u;
  const unsigned a = k < 0 ? 0u - unsigned(k) : unsigned(k);
  const int e = 31 - __clz(a | 1u);
  const unsigned long long m = (static_cast<unsigned long long>(a) << (52 - e)) & 0xFFFFFFFFFFFFFull;
  const unsigned long long bits =
      (static_cast<unsigned long long>(s) << 32) | (static_cast<unsigned long long>(1023 + e) << 52) | m;
  return k == 0 ? 0.0 : __longlong_as_double(static_cast<long long>(bits));
}
// Dequantized value k * q.
template <typename TS>
__device__ __forceinline__ TS dequant(int k, TS q) {
  return code_value<TS>(k) * q;
}

// One axis of a level in "slots".  Coarse node q (level node p(q) = min(2q,
// n-1)) owns two slots: its own, and the fine node p(q)+1 between q and q+1
// when there is one.  The plan tabulates per coarse node the five weights of
// its mass-transfer row on the slots (q-1).own, (q-1).fine, q.own, q.fine,
// (q+1).own -- 0 where a slot does not exist -- and the interpolation weights
// of q.fine (kSlot entries per node, filled by build_plan_tables).  In slots an
// axis of even length, whose last two nodes are both coarse, and the ends of
// an axis need no code of their own: their missing slots carry weight 0.
constexpr int kSlotWa = 5, kSlotWb = 6;  // entries 0..4: the row's weights

template <typename TS, typename TW>
struct LevelArgs {
  const void* in;  // DEC: level-l values (unit stride); REC: coefficients (nodal full grid, or the packed class)
  int64_t in_sz, in_sy;
  void* y;         // DEC: nodal output (full grid) or the packed class
  int64_t y_sz, y_sy;
  TW* w;           // DEC: coarse nodal values (compact m grid)
  TW* f;           // load vector (compact m grid)
  int64_t c_sz, c_sy;
  int n[3], m[3];
  int64_t s[3], N[3];   // full-grid map of a level-l node: min(i * s, N - 1)
  const TS* slot[3];    // slot tables, kSlot entries per coarse node
  int rows;        // coarse rows per strip
  int qz_chunk;    // coarse planes per z chunk
  int bz0;         // first z chunk of this launch (a launch may cover a subset of the chunks)
  int write_y;
  double qs;                // QZ: 1/bin width (MODE 0) or bin width (MODE 1)
  unsigned long long* qsat; // QZ, MODE 0: saturated-code counter (may be null)
  int all_fine;             // MODE 1: every node holds a coefficient (a time slice of a
                            // 4D field that is fine in time), not only the fine ones
};

// Units in flight per warp: a ring of units' rows in shared memory, filled by
// asynchronous copies all but one ahead.  Two units in FP64, whose units take
// over 3000 cycles of the FP64 pipe each, four in FP32.
template <typename TS>
constexpr int level_ring() {
  return sizeof(TS) == 8 ? 2 : 4;
}
// Row entries of a warp's y slot table: the rows of the strips its lanes can
// belong to and two before them.
__host__ __device__ inline int level_slot_rows(int mx, int my, int rows) {
  const int strips = (my + rows - 1) / rows, span = 31 / mx + 2;
  return (span < strips ? span : strips) * rows + 2;
}
// xy interpolants of a coarse plane that a lane keeps per unit.  FP64: four (both
// columns of the coarse row and of the fine row above it).  FP32 keeps the
// coarse row's two and forms the fine row's again from them (two FMAs and two
// products; the smaller footprint lets 16 instead of 12 warps reside on an SM),
// but for quantized output, whose fine rows have a rounding of their own.
template <int MODE, typename TS, bool QZ>
constexpr int level_interpolants() {
  return MODE == 1 ? 0 : (sizeof(TS) == 4 && !QZ) ? 2 : 4;
}
// Shared memory of one warp: the ring (four rows of 32 column pairs a unit), per
// unit (a strip of `rows` coarse rows has rows + 2) and lane the z accumulators
// of two coarse planes and the interpolants of the last one, and the y slots of
// its rows.
template <int MODE, typename TI, typename TS, bool QZ = false>
__host__ __device__ constexpr size_t level_smem_bytes(int rows, int slot_rows) {
  return sizeof(TI) * level_ring<TS>() * 256 +
         sizeof(TS) * (size_t(rows + 2) * 32 * (2 + level_interpolants<MODE, TS, QZ>()) + size_t(slot_rows) * kSlot);
}

// Lane groups of LX lanes over the coarse nodes of all strips of a level (strip
// by strip, each mx long): group g holds positions g*(LX-2) .. g*(LX-2)+LX-1,
// its first and last lanes only as neighbours.
template <int LX>
__host__ __device__ inline int64_t level_groups(int mx, int my, int rows) {
  const int64_t total = int64_t((my + rows - 1) / rows) * mx;
  return total <= LX ? 1 : (total - 2 + LX - 3) / (LX - 2);
}
template <int LX>
__host__ __device__ inline int64_t level_warps(int mx, int my, int rows) {
  return (level_groups<LX>(mx, my, rows) + 32 / LX - 1) / (32 / LX);
}

template <typename TS>
struct Slots {
  TS k0, k1, k2, k3, k4, wa, wb;
};
template <typename TS>
__device__ __forceinline__ Slots<TS> load_slots(const TS* t, int q);
template <>
__device__ __forceinline__ Slots<float> load_slots<float>(const float* t, int q) {
  const float4* p = reinterpret_cast<const float4*>(t) + 2 * q;
  const float4 a = p[0], b = p[1];
  return Slots<float>{a.x, a.y, a.z, a.w, b.x, b.y, b.z};
}
template <>
__device__ __forceinline__ Slots<double> load_slots<double>(const double* t, int q) {
  const double2* p = reinterpret_cast<const double2*>(t) + 4 * q;
  const double2 a = p[0], b = p[1], c = p[2], d = p[3];
  return Slots<double>{a.x, a.y, b.x, b.y, c.x, c.y, d.x};
}

// Values of the coarse and the fine plane of a pair: FP32 runs both planes'
// stencils as paired FMAs (per plane the same operations as scalar ones).
template <typename TS>
struct Planes {
  TS c, f;
};
// Five-tap sum in slot order, of both planes (HF) or of the coarse plane alone.
template <bool HF>
__device__ __forceinline__ Planes<double> taps(const Slots<double>& w, Planes<double> a, Planes<double> b,
                                               Planes<double> c, Planes<double> d, Planes<double> e) {
  Planes<double> r;
  r.c = fma(w.k4, e.c, fma(w.k3, d.c, fma(w.k2, c.c, fma(w.k1, b.c, w.k0 * a.c))));
  r.f = HF ? fma(w.k4, e.f, fma(w.k3, d.f, fma(w.k2, c.f, fma(w.k1, b.f, w.k0 * a.f)))) : 0.0;
  return r;
}
template <bool HF>
__device__ __forceinline__ Planes<float> taps(const Slots<float>& w, Planes<float> a, Planes<float> b,
                                              Planes<float> c, Planes<float> d, Planes<float> e) {
  if constexpr (HF) {
    float2 g = __fmul2_rn(make_float2(w.k0, w.k0), make_float2(a.c, a.f));
    g = __ffma2_rn(make_float2(w.k1, w.k1), make_float2(b.c, b.f), g);
    g = __ffma2_rn(make_float2(w.k2, w.k2), make_float2(c.c, c.f), g);
    g = __ffma2_rn(make_float2(w.k3, w.k3), make_float2(d.c, d.f), g);
    g = __ffma2_rn(make_float2(w.k4, w.k4), make_float2(e.c, e.f), g);
    return Planes<float>{g.x, g.y};
  } else {
    return Planes<float>{fmaf(w.k4, e.c, fmaf(w.k3, d.c, fmaf(w.k2, c.c, fmaf(w.k1, b.c, w.k0 * a.c)))), 0.f};
  }
}
template <int LX, bool HF, typename TS>
__device__ __forceinline__ Planes<TS> from_left(Planes<TS> v) {
  return Planes<TS>{__shfl_up_sync(0xffffffffu, v.c, 1, LX), HF ? __shfl_up_sync(0xffffffffu, v.f, 1, LX) : TS(0)};
}
template <int LX, bool HF, typename TS>
__device__ __forceinline__ Planes<TS> from_right(Planes<TS> v) {
  return Planes<TS>{__shfl_down_sync(0xffffffffu, v.c, 1, LX), HF ? __shfl_down_sync(0xffffffffu, v.f, 1, LX) : TS(0)};
}

// One warp's work: lane groups bx*32/LX .. and z chunk bz of level args `a`.
// PK: coefficients in the class-packed layout (MODE 0 writes `y`, MODE 1 reads
// `in` as the class of this level; y_sz / in_sz = n1*n2, y_sy / in_sy = n2).
// QZ (with PK): those coefficients are int32 codes (TD = int in MODE 0, TI =
// int in MODE 1).
// S1: the coefficients lie at unit stride (the finest level of the nodal layout;
// always when packed).
// AF: honour `all_fine` (the 4D form's time slices; a runtime flag read once).
template <int MODE, typename TI, typename TD, typename TS, typename TW, bool S1, bool PK = false, bool QZ = false,
          bool AF = false, int LX = 32>
__device__ __forceinline__ void level_body(const LevelArgs<TS, TW>& a, int bx, int bz, unsigned char* smem_raw) {
  static_assert(LX == 32 || LX == 16, "lane groups of a warp or half a warp");
  static_assert(S1 || !PK, "a packed class has unit stride");
  using TS2 = typename Pair<TS>::type;
  using TI2 = typename Pair<TI>::type;
  using P = Planes<TS>;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int IPN = level_interpolants<MODE, TS, QZ>(), RING = level_ring<TS>();
  // unit-stride input columns: the level's values (MODE 0), or unit-stride coefficients
  constexpr bool U1 = MODE == 0 || S1;
  // FP32 also computes what the first two units of a plane leave unused, instead
  // of branching around it; FP64, bound by its pipe, skips it
  constexpr bool SKIP = sizeof(TS) == 8;
  const int lid = threadIdx.x & 31, lane = lid % LX;
  const int nz = a.n[0], ny = a.n[1], nx = a.n[2];
  const int mz = a.m[0], my = a.m[1], mx = a.m[2];
  const int rows = a.rows;
  const int total = ((my + rows - 1) / rows) * mx;
  const int group = bx * (32 / LX) + lid / LX;
  const int pos = group * (LX - 2) + lane;
  const bool out = pos < total && (lane > 0 || group == 0) && (lane < LX - 1 || pos == total - 1);
  const int strip = min(pos, total - 1) / mx;
  const int q = min(pos, total - 1) - strip * mx;
  const int qy0 = strip * rows;
  const int nrow = min(rows, my - qy0);
  const int units = __reduce_max_sync(FULL, nrow) + 2;
  const int qz0 = bz * a.qz_chunk, qz1 = min(qz0 + a.qz_chunk, mz);
  const int t_start = max(qz0 - 1, 0), t_end = min(qz1, mz - 1);

  const TI* __restrict__ in = static_cast<const TI*>(a.in);
  TD* __restrict__ yout = static_cast<TD*>(a.y);
  // bounds-checking builds: extents (elements) of the buffers this warp
  // addresses; the LVL_* forms below check against them (other builds run the
  // plain accesses)
#ifdef MGR_DEBUG_BOUNDS
  const long long n_in = MODE == 0 ? (long long)nz * a.in_sz
                         : PK      ? (long long)nz * a.in_sz - (long long)mz * a.c_sz
                                   : (long long)a.N[0] * a.in_sz;
  const long long n_y = PK ? (long long)nz * a.y_sz - (long long)mz * a.c_sz : (long long)a.N[0] * a.y_sz;
  const long long n_c = (long long)mz * a.c_sz;
#endif
#define LVL_CP(dst, src) \
  MGR_GUARD(MGR_PIN(src, in, n_in, kDbgLevelIn) && MGR_PIN(dst, ring, RING * 256, kDbgLevelStage), \
            cp_async(dst, src, int(sizeof(TI))))
#define LVL_Y(p, v) MGR_GUARD(MGR_PIN(p, yout, n_y, kDbgLevelY), *(p) = (v))
#define LVL_W(p, v) MGR_GUARD(MGR_PIN(p, a.w, n_c, kDbgLevelW), *(p) = (v))
#define LVL_F(p, v) MGR_GUARD(MGR_PIN(p, a.f, n_c, kDbgLevelF), *(p) = (v))
  const bool afine = AF && MODE == 1 && a.all_fine;
  const TS qs = QZ ? TS(a.qs) : TS(1);
  // value written for coefficient v (MODE 0); value of a read coefficient
  // (MODE 1; with QZ the code itself: the bin width scales the load vector
  // once per coarse node instead, see fout)
  auto yval = [&](TS v) -> TD {
    if constexpr (QZ) return TD(quant_code(v, qs, a.qsat));
    else return TD(v);
  };
  auto cval = [&](TI v) -> TS {
    if constexpr (QZ && MODE == 1) return code_value<TS>(int(v));
    else return TS(v);
  };
  auto fout = [&](TS acc) -> TW {
    if constexpr (QZ && MODE == 1) return TW(acc) * TW(a.qs);
    else return TW(acc);
  };

  // ---- this lane's column: own node and, when fx, the fine node after it
  const Slots<TS> kx = load_slots<TS>(a.slot[2], q);
  const bool fx = 2 * q + 1 < nx - 1;
  // input columns.  Unit stride: the pair (c, c+1), c = 2q; the axis' last node
  // has no right neighbour and reads (n-2, n-1), its own value second (swp).
  // Strided: own node, and the fine node or, where there is none, the own node
  // again.  A slot without a node holds some value of the row and meets weight 0.
  const bool swp = U1 && 2 * q >= nx - 1;
  const int ic0 = U1 ? min(2 * q, nx - 2) : int(min(2 * int64_t(q) * a.s[2], a.N[2] - 1));
  const int64_t icd = U1 ? 1 : (fx ? a.s[2] : 0);
  // output columns (MODE 0)
  const int yc0 = PK ? min(2 * q, nx - 1) : int(min(2 * int64_t(q) * a.s[2], a.N[2] - 1));
  const int64_t ycd = S1 ? 1 : a.s[2];
  // rows of the level (see StripRows), in (r) the input and (o) the output
  const int rs = U1 ? 1 : int(a.s[1]), rN = U1 ? ny : int(a.N[1]), isy = int(a.in_sy);
  const int os = S1 ? 1 : int(a.s[1]), oN = S1 ? ny : int(a.N[1]), ysy = int(a.y_sy);
  const int csy = int(a.c_sy);

  // z plane offsets (in: level plane g; coarse planes are g = p(t))
  auto iplane = [&](int g) -> int64_t {
    if (PK && MODE == 1) return int64_t(g) * a.in_sz - int64_t(cidx(g)) * a.c_sz;
    return U1 ? int64_t(g) * a.in_sz : fmap(g, a.s[0], a.N[0]) * a.in_sz;
  };
  auto yplane = [&](int g) -> int64_t {
    if (PK) return int64_t(g) * a.y_sz - int64_t(cidx(g)) * a.c_sz;
    return S1 ? int64_t(g) * a.y_sz : fmap(g, a.s[0], a.N[0]) * a.y_sz;
  };
  auto has_fine = [&](int t) { return t > t_start && pidx(t, nz) - pidx(t - 1, nz) == 2; };

  // ---- shared memory: ring, z accumulators, interpolants, y slots
  TI* ring = reinterpret_cast<TI*>(smem_raw);                               // [ring][4 rows][own, fine column][32 lanes]
  TS* acc_s = reinterpret_cast<TS*>(ring + RING * 256);               // [units][32][2]
  TS* ip_s = acc_s + (rows + 2) * 64;                                       // [units][32][IPN]
  TS* ky_s = ip_s + (rows + 2) * 32 * IPN;                                  // [slot rows][kSlot]
  {
    // rows qy0 - 2 of the first lane's strip on; rows outside the grid have weights 0
    const int first_row = __shfl_sync(FULL, qy0, 0) - 2, n = level_slot_rows(mx, my, rows);
    for (int i = lid; i < n * kSlot; i += 32) {
      const int row = first_row + i / kSlot;
      ky_s[i] = (row >= 0 && row < my) ? a.slot[1][int64_t(row) * kSlot + i % kSlot] : TS(0);
    }
    __syncwarp();
    ky_s += (qy0 - 2 - first_row) * kSlot;  // this lane's unit 0
  }

  // ---- copies of the next unit (unit lu of plane pair lt) into the ring slot at
  // d0 / d1 (own / fine column).  Rows cr, cs, fr, fs: the coarse row p(qc) and
  // the fine row above it, in the coarse plane and the fine plane; rows outside
  // the grid read some row of it and carry weight 0
  int lt = t_start, lu = 0, lslot = 0;
  StripRows lrow(qy0, rs, rN, isy);
  bool lhf = false;
  const TI *lc = nullptr, *lf = nullptr;
  auto load_planes = [&]() {
    const int p = pidx(lt, nz);
    lhf = has_fine(lt);
    lc = in + iplane(p) + ic0;
    lf = lhf ? in + iplane(p - 1) + ic0 : lc;
  };
  TI* const ring0 = ring + lid + (swp ? 32 : 0);
  TI* const ring1 = ring + lid + (swp ? 0 : 32);
  auto load_unit = [&]() {
    if (lt <= t_end) {
      TI* d0 = ring0 + lslot * 256;
      TI* d1 = ring1 + lslot * 256;
      TI* dx = ring + lslot * 256 + lid + 32;  // the fine column's slot
      // element offsets of the two rows, clamped into the plane
      const int r = lrow.coarse(), s = lrow.fine();
      lrow.next(lu == 0);
      if constexpr (PK && MODE == 1) {
        // rows of a coarse plane: the coarse row holds its fine columns only
        // (slots without a value: 0, they meet weights 0)
        const int qc = min(max(qy0 - 1 + lu, 0), my - 1);
        if (fx && qy0 - 1 + lu == qc) LVL_CP(dx, lc - ic0 + (r - qc * mx + q));
        else *dx = TI(0);
        if (2 * qc - 1 < ny - 1 && qc > 0) {
          const int o = (2 * qc - 1) * nx - qc * mx;
          LVL_CP(d0 + 64, lc + o);
          LVL_CP(d1 + 64, lc + o + 1);
        } else {
          d0[64] = d1[64] = TI(0);
        }
        if (lhf) {
          LVL_CP(d0 + 128, lf + r);
          LVL_CP(d1 + 128, lf + r + 1);
          LVL_CP(d0 + 192, lf + s);
          LVL_CP(d1 + 192, lf + s + 1);
        }
      } else {
        const TI *pr = lc + r, *ps = lc + s;
        if (MODE == 0 || AF) {
          LVL_CP(d0, pr);
          LVL_CP(d1, pr + icd);
        } else {
          LVL_CP(dx, swp ? pr : pr + icd);  // (the own column holds no coefficient)
        }
        if (!SKIP || lu > 0) {
          LVL_CP(d0 + 64, ps);
          LVL_CP(d1 + 64, ps + icd);
        }
        if (lhf) {
          const TI *fr = lf + r, *fs = lf + s;
          LVL_CP(d0 + 128, fr);
          LVL_CP(d1 + 128, fr + icd);
          if (!SKIP || lu > 0) {
            LVL_CP(d0 + 192, fs);
            LVL_CP(d1 + 192, fs + icd);
          }
        }
      }
      lslot = (lslot + 1) & (RING - 1);
      if (++lu == units) {
        lu = 0;
        lrow.restart();
        ++lt;
        if (lt <= t_end) load_planes();
      }
    }
    cp_commit();
  };
  load_planes();
#pragma unroll
  for (int i = 0; i < RING - 1; ++i) load_unit();
  int slot = 0;  // ring slot of the unit being processed
  // (QZ, FP32) parity of qc below the fine rows with the other rounding: row pairs
  // count from the one before the 14-row strip that this strip is part of, from
  // its first one in the first of them, and from two before where it starts on
  // the last node of an axis of even length
  const int qy14 = qy0 - qy0 % 14;
  const int qz_parity = (qy14 + ((qy14 == 0 || (qy14 == my - 1 && (ny & 1) == 0)) ? 0 : 1)) & 1;
  // rows with outputs, by unit: coarse rows u - 1 < nr, fine rows u - 2 < ns, all
  // 0 on lanes without outputs
  const unsigned nr = out ? nrow : 0, ns = out ? min(nrow, max((ny - 1) / 2 - qy0, 0)) : 0;
  const unsigned nrx = fx ? nr : 0, nsx = fx ? ns : 0;  // at the fine column

  // ---- one plane pair (HF: with a fine plane)
  auto plane_pair = [&](auto hf_c, int t) {
    constexpr bool HF = decltype(hf_c)::value;
    const int Pc = pidx(t, nz);
    const bool own_c = t >= qz0 && t < qz1, own_f = HF && t > qz0;
    const bool wy_c = own_c && a.write_y, wy_f = own_f && a.write_y;  // coefficients written
    TD* yzc = MODE == 0 ? yout + yplane(Pc) + yc0 : nullptr;
    TD* yzf = MODE == 0 ? yout + yplane(HF ? Pc - 1 : Pc) + yc0 : nullptr;
    // coarse values of this plane and load vector of the plane before it, at the unit's row
    TW* wp = MODE == 0 ? a.w + (int64_t(t) * a.c_sz + (int64_t(qy0) - 1) * csy + q) : nullptr;
    TW* fp = a.f + (int64_t(t - 1) * a.c_sz + (int64_t(qy0) - 2) * csy + q);
    const unsigned nf = (t - 1 >= qz0 && t - 1 < qz1) ? nr : 0;       // plane t-1 complete
    const unsigned nl = (t == mz - 1 && t < qz1) ? nr : 0;            // the last plane, too
    // z weights of the two planes for the coarse planes t-1, t, t+1, and of the fine plane's interpolant
    const TS* zt = a.slot[0] + int64_t(kSlot) * t;
    const TS wzc0 = t > 0 ? zt[4 - kSlot] : TS(0), wzf0 = HF ? zt[3 - kSlot] : TS(0);
    const TS wzc1 = zt[2], wzf1 = HF ? zt[1] : TS(0);
    const TS wzc2 = t + 1 < mz ? zt[kSlot] : TS(0);
    const TS za = (MODE == 0 && HF) ? zt[kSlotWa - kSlot] : TS(0), zb = (MODE == 0 && HF) ? zt[kSlotWb - kSlot] : TS(0);
    const bool first = t == t_start;

    // x-stencil results of the rows before: (qc-2).own, (qc-2).fine, (qc-1).own
    P ga{}, gb{}, gc{};
    TS i0p = TS(0), i1p = TS(0);  // x interpolants of coarse row qc-1 in this plane
    TS j0p = TS(0), j1p = TS(0);  // and in the coarse plane before (IPN == 2)
    int qc = qy0 - 1;
    TS* ip = ip_s + lid * IPN;
    TS2* ap = reinterpret_cast<TS2*>(acc_s + lid * 2);
    const TS* kp = ky_s;
    StripRows orow(qy0, os, oN, ysy);  // output rows
    orow.rewind();
#pragma unroll 2
    for (int u = 0; u < units; ++u, ++qc) {
      // each lane copies, and reads, only its own slots of the ring
      load_unit();
      cp_wait<RING - 1>();
      const TI* d = ring + slot * 256 + lid;
      slot = (slot + 1) & (RING - 1);
      const TI2 vcr{d[0], d[32]}, vcs{d[64], d[96]};
      TI2 vfr{}, vfs{};
      if constexpr (HF) {
        vfr = TI2{d[128], d[160]};
        vfs = TI2{d[192], d[224]};
      }
      // weights of coarse row qc-1: its stencil row and its fine row's interpolation
      const Slots<TS> ky = load_slots<TS>(kp, 0);
      kp += kSlot;

      // ---- coefficients, own (0) and fine (1) column: coarse row (r), fine row above it (s)
      P r0{}, r1{}, s0{}, s1{};
      if constexpr (MODE == 0) {
        const TS v0 = cval(vcr.x);
        const TS vr = __shfl_down_sync(FULL, v0, 1, LX);
        const TS i0 = v0;
        TS i1 = fx ? fma(kx.wb, vr, kx.wa * v0) : TS(0);
        TS i1n = i1;  // as the lower neighbour of the fine row
        if constexpr (QZ && sizeof(TS) == 4) {
          // FP32 codes are whole numbers that show the last bit of a coefficient, and
          // they keep the values they have always had: there the interpolant was
          // rounded the other way round on the last row of an axis of even length
          // and below every second fine row of a strip of 14
          const TS other = fx ? fma(kx.wa, v0, kx.wb * vr) : TS(0);
          if (qc == my - 1 && (ny & 1) == 0) i1 = other;
          if ((qc & 1) == qz_parity) i1n = other;
        }
        const TS i2 = fma(ky.wa, i0p, ky.wb * i0), i3 = fma(ky.wa, i1p, ky.wb * i1n);
        r1.c = cval(vcr.y) - i1;
        s0.c = cval(vcs.x) - i2;
        s1.c = cval(vcs.y) - i3;
        if constexpr (IPN == 2) {
          if constexpr (HF) {
            const float2 p = *reinterpret_cast<const float2*>(ip);
            const TS p2 = fma(ky.wa, j0p, ky.wb * p.x), p3 = fma(ky.wa, j1p, ky.wb * p.y);
            r0.f = cval(vfr.x) - za * p.x - zb * i0;
            r1.f = cval(vfr.y) - za * p.y - zb * i1;
            s0.f = cval(vfs.x) - za * p2 - zb * i2;
            s1.f = cval(vfs.y) - za * p3 - zb * i3;
            j0p = p.x;
            j1p = p.y;
          }
          *reinterpret_cast<float2*>(ip) = make_float2(i0, i1);
        } else {
          if constexpr (HF) {
            const TS2 p = *reinterpret_cast<const TS2*>(ip), pp = *reinterpret_cast<const TS2*>(ip + 2);
            r0.f = cval(vfr.x) - za * p.x - zb * i0;
            r1.f = cval(vfr.y) - za * p.y - zb * i1;
            s0.f = cval(vfs.x) - za * pp.x - zb * i2;
            s1.f = cval(vfs.y) - za * pp.y - zb * i3;
          }
          *reinterpret_cast<TS2*>(ip) = TS2{i0, i1};
          *reinterpret_cast<TS2*>(ip + 2) = TS2{i2, i3};
        }
        ip += 32 * IPN;
        i0p = i0;
        i1p = i1;
      } else {
        // where the coarse plane has no fine column or fine row, its slots hold
        // values of coarse nodes, which may be infinite: 0, not only weight 0
        const bool fine_row = qc > 0 && 2 * qc - 1 < ny - 1;
        r0.c = afine ? cval(vcr.x) : TS(0);
        r1.c = fx ? cval(vcr.y) : TS(0);
        s0.c = fine_row ? cval(vcs.x) : TS(0);
        s1.c = fine_row ? cval(vcs.y) : TS(0);
        if constexpr (HF) {
          r0.f = cval(vfr.x);
          r1.f = cval(vfr.y);
          s0.f = cval(vfs.x);
          s1.f = cval(vfs.y);
        }
      }

      // ---- coefficient and coarse-value outputs
      if constexpr (MODE == 0) {
        const unsigned ur = unsigned(u - 1), us = unsigned(u - 2);
        const bool wr = ur < nr, wrx = ur < nrx, ws = us < ns, wsx = us < nsx;
        const int oc = orow.coarse(), osr = orow.above();
        orow.advance();
        if (own_c && wr) LVL_W(wp, TW(vcr.x));
        wp += csy;
        if (wy_c) {
          if constexpr (PK) {
            // rows of a coarse plane leave the coarse nodes out: the coarse row keeps its fine columns
            const int out_c = qc * mx;
            if (wrx) LVL_Y(yzc + (oc - out_c + q - yc0), yval(r1.c));
            if (ws) LVL_Y(yzc + (osr - out_c), yval(s0.c));
            if (wsx) LVL_Y(yzc + (osr - out_c) + 1, yval(s1.c));
          } else {
            // (all-coarse nodes get a placeholder that a coarser level overwrites:
            // at unit stride it keeps the row's sectors fully written)
            TD *pr = yzc + oc, *ps = yzc + osr;
            if (S1 && wr) LVL_Y(pr, TD(0));
            if (wrx) LVL_Y(pr + ycd, TD(r1.c));
            if (ws) LVL_Y(ps, TD(s0.c));
            if (wsx) LVL_Y(ps + ycd, TD(s1.c));
          }
        }
        if (HF && wy_f) {
          TD *pr = yzf + oc, *ps = yzf + osr;
          if (wr) LVL_Y(pr, yval(r0.f));
          if (wrx) LVL_Y(pr + ycd, yval(r1.f));
          if (ws) LVL_Y(ps, yval(s0.f));
          if (wsx) LVL_Y(ps + ycd, yval(s1.f));
        }
      }

      // ---- x stencil of the unit's rows (the coefficients of the coarse plane's
      // coarse row vanish on coarse nodes)
      P gd{}, ge;
      if (!SKIP || u > 0) gd = taps<HF>(kx, from_left<LX, HF>(s0), from_left<LX, HF>(s1), s0, s1, from_right<LX, HF>(s0));
      if constexpr (sizeof(TS) == 8) {
        const P l1 = from_left<LX, HF>(r1);
        if (AF && afine) {
          ge = taps<HF>(kx, from_left<LX, HF>(r0), l1, r0, r1, from_right<LX, HF>(r0));
        } else {
          ge.c = fma(kx.k3, r1.c, kx.k1 * l1.c);
          ge.f = HF ? fma(kx.k4, __shfl_down_sync(FULL, r0.f, 1, LX),
                          fma(kx.k3, r1.f, fma(kx.k2, r0.f, fma(kx.k1, l1.f, kx.k0 * __shfl_up_sync(FULL, r0.f, 1, LX)))))
                    : TS(0);
        }
      } else {
        P l0{}, e0{};
        if (AF && afine) {
          l0 = from_left<LX, HF>(r0);
          e0 = from_right<LX, HF>(r0);
        } else if constexpr (HF) {
          l0.f = __shfl_up_sync(FULL, r0.f, 1, LX);
          e0.f = __shfl_down_sync(FULL, r0.f, 1, LX);
        }
        ge = taps<HF>(kx, l0, from_left<LX, HF>(r1), r0, r1, e0);
      }

      // ---- y stencil of coarse row qc-1 and its z accumulation
      if (!SKIP || u > 1) {
        TS2 acc = *ap;
        if (first) acc.x = acc.y = TS(0);
        const P g = taps<HF>(ky, ga, gb, gc, gd, ge);
        acc.x = fma(wzc0, g.c, acc.x);
        acc.y = fma(wzc1, g.c, acc.y);
        const TS a2 = wzc2 * g.c;
        if constexpr (HF) {
          acc.x = fma(wzf0, g.f, acc.x);
          acc.y = fma(wzf1, g.f, acc.y);
        }
        *ap = TS2{acc.y, a2};
        if (unsigned(u - 2) < nf) LVL_F(fp, fout(acc.x));
        if (unsigned(u - 2) < nl) LVL_F(fp + a.c_sz, fout(acc.y));
      }
      ap += 32;
      fp += csy;
      ga = gc;
      gb = gd;
      gc = ge;
    }
  };
  for (int t = t_start; t <= t_end; ++t) {
    if (has_fine(t)) plane_pair(std::true_type{}, t);
    else plane_pair(std::false_type{}, t);
  }
}

#undef LVL_CP
#undef LVL_Y
#undef LVL_W
#undef LVL_F

// Warps per SM the pass is compiled for: 16 (128 registers a thread), but 12 (168) for
// the FP64 decomposition.
template <int MODE, typename TS>
constexpr int level_ctas() {
  return MODE == 0 && sizeof(TS) == 8 ? 12 : 16;
}

template <int MODE, typename TI, typename TD, typename TS, typename TW, bool S1, bool PK, bool QZ>
__global__ void __launch_bounds__(32, level_ctas<MODE, TS>()) k_level(const LevelArgs<TS, TW> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  level_body<MODE, TI, TD, TS, TW, S1, PK, QZ>(a, blockIdx.x, blockIdx.y + a.bz0, smem_raw);
}

// ---------------------------------------------------------------------------
// Recomposition interpolation (Sec. II.A, recomposition): level-l values
// v = c + (P_z x P_y x P_x) v_coarse, in the level pass's units: one warp takes a
// strip of coarse rows and a chunk of coarse planes for the coarse x nodes of its
// lanes, plane pair by plane pair (the coarse plane t and the fine plane before
// it), each in units of the coarse row qc and the fine row above it.  A lane
// reads its right neighbour's coarse value itself, so every lane of a warp has
// outputs, whatever the width (tiles 32 nodes wide took 9 tiles, 288 lanes, for
// 257 nodes).  The strip's row before the first and the chunk's plane before the
// first are interpolated only.  The x interpolants of the previous row stay in
// registers, the xy interpolants of the previous plane in the lane's own
// shared-memory slots; coefficients and coarse values arrive in a ring of units
// by asynchronous copies three units ahead.  No step waits for another warp.
// The output lies at unit stride (the field, or a compact level).
// What bounds it: FP64 the FP64 pipe (17 operations of 16 cycles a unit), FP32
// memory (its reads and writes at 0.77 of the copy rate).  513^3, finest level,
// against 256-thread CTAs over 32 x 16 tiles: FP64 0.721 -> 0.582 ms, FP32 0.219 ->
// 0.225 ms (the writes of neighbouring warps merge less), 257^3 FP32 0.047 -> 0.039
// ms, 129^3 FP64 0.036 -> 0.025 ms; 1501 coarse columns of a plane 22 -> 16 us.
// ---------------------------------------------------------------------------
template <typename TS, typename TW>
struct InterpArgs {
  const void* c;  // coefficients: nodal (full grid) or this level's packed class; null = all zero
  int64_t y_sz, y_sy;
  const TW* w;    // coarse values (compact m grid)
  int64_t c_sz, c_sy;
  void* out;      // level-l values
  int64_t o_sz, o_sy;
  int n[3], m[3];
  int64_t s[3], N[3];
  const TS* slot[3];
  int rows;       // coarse rows per strip
  int qz_chunk;   // coarse planes per z chunk
  int bz0;        // first z chunk of this launch (a launch may cover a subset of the chunks)
  double qs;      // QZ: bin width of the level's class
};

constexpr int kInterpRing = 4;  // units in flight per warp
// Warps over the coarse nodes of all strips, 32 each.
__host__ __device__ inline int64_t interp_warps(int mx, int my, int rows) {
  return (int64_t((my + rows - 1) / rows) * mx + 31) / 32;
}
// Shared memory of one warp: the ring (seven coefficients and two coarse values a
// lane and unit), per unit and lane the four xy interpolants of the last coarse
// plane, and the y interpolation weights of its rows.
template <typename TD, typename TS, typename TW>
__host__ __device__ constexpr size_t interp_smem_bytes(int rows, int slot_rows) {
  return kInterpRing * 32 * (7 * sizeof(TD) + 2 * sizeof(TW)) +
         sizeof(TS) * (size_t(rows + 1) * 32 * 4 + size_t(slot_rows) * 2);
}

// One warp's work: positions 32 bx .. of the strips' nodes and z chunk bz.
// PK: `c` is the class-packed class of this level (y_sz = n1*n2, y_sy = n2).
// QZ (with PK): `c` holds int32 codes (TD = int), coefficient = code * qs.
// S1: the coefficients lie at unit stride (the finest level, or packed).
template <typename TD, typename TO, typename TS, typename TW, bool S1, bool PK = false, bool QZ = false>
__device__ __forceinline__ void interp_body(const InterpArgs<TS, TW>& a, int bx, int bz, unsigned char* smem_raw) {
  static_assert(S1 || !PK, "a packed class has unit stride");
  using TS2 = typename Pair<TS>::type;
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int RING = kInterpRing;
  const int lid = threadIdx.x & 31;
  const int nz = a.n[0], ny = a.n[1], nx = a.n[2];
  const int mz = a.m[0], my = a.m[1], mx = a.m[2];
  const int rows = a.rows;
  const int total = ((my + rows - 1) / rows) * mx;
  const bool out_lane = bx * 32 + lid < total;
  const int pos = min(bx * 32 + lid, total - 1);
  const int strip = pos / mx, q = pos - strip * mx;
  const int qy0 = strip * rows;
  const int nrow = min(rows, my - qy0);
  const int units = __reduce_max_sync(FULL, nrow) + 1;
  const int qz0 = bz * a.qz_chunk, qz1 = min(qz0 + a.qz_chunk, mz);
  const int t_start = max(qz0 - 1, 0), t_end = qz1 - 1;

  const TD* __restrict__ cin = static_cast<const TD*>(a.c);
  const bool cz = cin == nullptr;  // coefficients of a dropped class: zero
  TO* __restrict__ out = static_cast<TO*>(a.out);
  // bounds-checking builds: extents of the buffers; the ITP_* forms check
  // against them (other builds run the plain accesses)
#ifdef MGR_DEBUG_BOUNDS
  const long long n_ci = PK ? (long long)nz * a.y_sz - (long long)mz * a.c_sz : (long long)a.N[0] * a.y_sz;
  const long long n_w = (long long)mz * a.c_sz;
  const long long n_o = (long long)nz * a.o_sz;
#endif
#define ITP_CP(dst, src)                                                                                           \
  MGR_GUARD(MGR_PIN(src, cin, n_ci, kDbgInterpC) && MGR_PIN(dst, ring, RING * 7 * 32, kDbgInterpStage), \
            cp_async(dst, src, int(sizeof(TD))))
#define ITP_CW(dst, src)                                                                                             \
  MGR_GUARD(MGR_PIN(src, a.w, n_w, kDbgInterpW) && MGR_PIN(dst, wring, RING * 2 * 32, kDbgInterpStage), \
            cp_async(dst, src, int(sizeof(TW))))
#define ITP_O(p, v) MGR_GUARD(MGR_PIN(p, out, n_o, kDbgInterpOut), *(p) = (v))
  const TS qs = QZ ? TS(a.qs) : TS(1);
  // coefficient v plus interpolant b (QZ: code * q + b in one FMA)
  auto cadd = [&](TD v, TS b) -> TS {
    if constexpr (QZ) return fma(code_value<TS>(int(v)), qs, b);
    else return TS(v) + b;
  };
  // coefficient v plus the interpolant between the coarse planes' p and i
  auto zadd = [&](TD v, TS za, TS p, TS zb, TS i) -> TS {
    if constexpr (QZ) return cadd(v, za * p + zb * i);
    else return TS(v) + za * p + zb * i;
  };

  // ---- this lane's column (see level_body: slots, swapped pair at the end)
  const TS wax = a.slot[2][int64_t(kSlot) * q + kSlotWa], wbx = a.slot[2][int64_t(kSlot) * q + kSlotWb];
  const bool fx = 2 * q + 1 < nx - 1;
  const bool swp = S1 && 2 * q >= nx - 1;
  const int ic0 = S1 ? min(2 * q, nx - 2) : int(min(2 * int64_t(q) * a.s[2], a.N[2] - 1));
  const int64_t icd = S1 ? 1 : (fx ? a.s[2] : 0);
  const int wcd = q + 1 < mx ? 1 : 0;  // right neighbour's coarse value
  const int oc0 = min(2 * q, nx - 1);
  const int rs = S1 ? 1 : int(a.s[1]), rN = S1 ? ny : int(a.N[1]), isy = int(a.y_sy);
  const int osy = int(a.o_sy), csy = int(a.c_sy);
  auto cplane = [&](int g) -> int64_t {
    if (PK) return int64_t(g) * a.y_sz - int64_t(cidx(g)) * a.c_sz;
    return S1 ? int64_t(g) * a.y_sz : fmap(g, a.s[0], a.N[0]) * a.y_sz;
  };
  auto has_fine = [&](int t) { return t > t_start && pidx(t, nz) - pidx(t - 1, nz) == 2; };

  // ---- shared memory: rings, interpolants, y weights
  TD* ring = reinterpret_cast<TD*>(smem_raw);               // [ring][7][32]: r fine; s, fr, fs own and fine
  TW* wring = reinterpret_cast<TW*>(ring + RING * 7 * 32);  // [ring][2][32]: own, right neighbour
  TS* ip_s = reinterpret_cast<TS*>(wring + RING * 2 * 32);  // [units][32][4]
  TS* ky_s = ip_s + (rows + 1) * 128;                       // [slot rows][2]
  {
    // rows qy0 - 2 of the first lane's strip on; rows outside the grid have weights 0
    const int first_row = __shfl_sync(FULL, qy0, 0) - 2, n = level_slot_rows(mx, my, rows);
    for (int i = lid; i < n * 2; i += 32) {
      const int row = first_row + i / 2;
      ky_s[i] = (row >= 0 && row < my) ? a.slot[1][int64_t(row) * kSlot + kSlotWa + i % 2] : TS(0);
    }
    if (cz)
      for (int i = lid; i < RING * 7 * 32; i += 32) ring[i] = TD(0);
    __syncwarp();
    ky_s += (qy0 - 2 - first_row) * 2;  // this lane's unit 0
  }

  // ---- copies of the next unit (unit lu of plane pair lt)
  int lt = t_start, lu = 0, lslot = 0;
  StripRows lrow(qy0, rs, rN, isy);
  lrow.rewind();
  const int wrow0 = (qy0 - 1) * csy, wrow_max = (my - 1) * csy;
  int wrow = wrow0;
  bool lhf = false, lc_on = false;
  const TD *lc = nullptr, *lf = nullptr;
  const TW* lw = nullptr;
  auto load_planes = [&]() {
    const int p = pidx(lt, nz);
    lhf = !cz && has_fine(lt);
    lc_on = !cz && lt >= qz0;
    lw = a.w + (int64_t(lt) * a.c_sz + q);
    if (!cz) {
      lc = cin + cplane(p) + ic0;
      lf = lhf ? cin + cplane(p - 1) + ic0 : lc;
    }
  };
  auto load_unit = [&]() {
    if (lt <= t_end) {
      TW* dw = wring + lslot * 64 + lid;
      const TW* pw = lw + min(max(wrow, 0), wrow_max);
      ITP_CW(dw, pw);
      ITP_CW(dw + 32, pw + wcd);
      if (lu > 0) {
        TD* dx = ring + lslot * 224 + lid;              // fine column of the coarse row
        TD* d0 = dx + (swp ? 64 : 32);                  // own columns of the other rows
        TD* d1 = dx + (swp ? 32 : 64);                  // fine columns
        const int r = lrow.coarse(), s = lrow.above();
        if (lc_on) {
          if constexpr (PK) {
            // rows of a coarse plane: the coarse row holds its fine columns only
            const int qc = min(qy0 - 1 + lu, my - 1);
            if (fx && qy0 - 1 + lu == qc) ITP_CP(dx, lc - ic0 + (r - qc * mx + q));
            if (2 * qc - 1 < ny - 1 && qc > 0) {
              const int o = (2 * qc - 1) * nx - qc * mx;
              ITP_CP(d0, lc + o);
              ITP_CP(d1, lc + o + 1);
            }
          } else {
            const TD *pr = lc + r, *ps = lc + s;
            ITP_CP(dx, swp ? pr : pr + icd);
            ITP_CP(d0, ps);
            ITP_CP(d1, ps + icd);
          }
        }
        if (lhf) {
          const TD *fr = lf + r, *fs = lf + s;
          ITP_CP(d0 + 64, fr);
          ITP_CP(d1 + 64, fr + icd);
          ITP_CP(d0 + 128, fs);
          ITP_CP(d1 + 128, fs + icd);
        }
      }
      lslot = (lslot + 1) & (RING - 1);
      lrow.advance();
      wrow += csy;
      if (++lu == units) {
        lu = 0;
        lrow.rewind();
        wrow = wrow0;
        ++lt;
        if (lt <= t_end) load_planes();
      }
    }
    cp_commit();
  };
  load_planes();
#pragma unroll
  for (int i = 0; i < RING - 1; ++i) load_unit();
  int slot = 0;
  // rows with outputs, by unit: coarse rows u - 1 < nr, the fine rows above them where they exist
  const unsigned nr = out_lane ? nrow : 0, nrx = fx ? nr : 0;

  // ---- one plane pair (HF: with a fine plane)
  auto plane_pair = [&](auto hf_c, int t) {
    constexpr bool HF = decltype(hf_c)::value;
    const int Pc = pidx(t, nz);
    const bool own_c = t >= qz0;
    TO* ozc = out + (int64_t(Pc) * a.o_sz + oc0);
    TO* ozf = out + (int64_t(HF ? Pc - 1 : Pc) * a.o_sz + oc0);
    const TS* zt = a.slot[0] + int64_t(kSlot) * t;
    const TS za = HF ? zt[kSlotWa - kSlot] : TS(0), zb = HF ? zt[kSlotWb - kSlot] : TS(0);
    TS i0p = TS(0), i1p = TS(0);  // x interpolants of coarse row qc-1
    int qc = qy0 - 1;
    TS* ip = ip_s + lid * 4;
    const TS* kp = ky_s;
    StripRows orow(qy0, 1, ny, osy);
    orow.rewind();
#pragma unroll 2
    for (int u = 0; u < units; ++u, ++qc) {
      // each lane copies, and reads, only its own slots of the rings
      load_unit();
      cp_wait<RING - 1>();
      const TD* d = ring + slot * 224 + lid;
      const TW* dw = wring + slot * 64 + lid;
      slot = (slot + 1) & (RING - 1);
      const TW w0 = dw[0];
      const TS i0 = TS(w0), i1 = fx ? fma(wbx, TS(dw[32]), wax * i0) : TS(0);
      const TS2 ky = *reinterpret_cast<const TS2*>(kp);  // interpolation weights of the fine row above
      kp += 2;
      const TS i2 = fma(ky.x, i0p, ky.y * i0), i3 = fma(ky.x, i1p, ky.y * i1);
      TS2 p{}, pp{};
      if constexpr (HF) {
        if constexpr (sizeof(TS) == 4) {
          const float4 v = *reinterpret_cast<const float4*>(ip);
          p = TS2{v.x, v.y};
          pp = TS2{v.z, v.w};
        } else {
          p = *reinterpret_cast<const TS2*>(ip);
          pp = *reinterpret_cast<const TS2*>(ip + 2);
        }
      }
      if constexpr (sizeof(TS) == 4) {
        *reinterpret_cast<float4*>(ip) = make_float4(i0, i1, i2, i3);
      } else {
        *reinterpret_cast<TS2*>(ip) = TS2{i0, i1};
        *reinterpret_cast<TS2*>(ip + 2) = TS2{i2, i3};
      }
      ip += 128;
      i0p = i0;
      i1p = i1;
      const bool fine_row = 2 * qc - 1 < ny - 1 && qc > 0;
      const bool wr = unsigned(u - 1) < nr, wrx = unsigned(u - 1) < nrx;
      const bool ws = wr && fine_row, wsx = wrx && fine_row;
      const int oc = orow.coarse(), osr = orow.above();
      orow.advance();
      if (own_c && u > 0) {
        TO *pr = ozc + oc, *ps = ozc + osr;
        if (wr) ITP_O(pr, TO(w0));
        if (wrx) ITP_O(pr + 1, TO(cadd(d[0], i1)));
        if (ws) ITP_O(ps, TO(cadd(d[32], i2)));
        if (wsx) ITP_O(ps + 1, TO(cadd(d[64], i3)));
      }
      if (HF && u > 0) {
        TO *pr = ozf + oc, *ps = ozf + osr;
        if (wr) ITP_O(pr, TO(zadd(d[96], za, p.x, zb, i0)));
        if (wrx) ITP_O(pr + 1, TO(zadd(d[128], za, p.y, zb, i1)));
        if (ws) ITP_O(ps, TO(zadd(d[160], za, pp.x, zb, i2)));
        if (wsx) ITP_O(ps + 1, TO(zadd(d[192], za, pp.y, zb, i3)));
      }
    }
  };
  for (int t = t_start; t <= t_end; ++t) {
    if (has_fine(t)) plane_pair(std::true_type{}, t);
    else plane_pair(std::false_type{}, t);
  }
}

#undef ITP_CP
#undef ITP_CW
#undef ITP_O

template <typename TD, typename TO, typename TS, typename TW, bool S1, bool PK, bool QZ>
__global__ void __launch_bounds__(32, 16) k_interp(const InterpArgs<TS, TW> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  interp_body<TD, TO, TS, TW, S1, PK, QZ>(a, blockIdx.x, blockIdx.y + a.bz0, smem_raw);
}
