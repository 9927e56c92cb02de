// k_stencil2d_stream.cuh -- register-resident, warp-streamed time tiling of
// a 1-D / 2-D iterated stencil (any boundary rule).
//
// A warp owns a strip of 32*C consecutive columns (C per lane, one 16-byte
// vector) and streams down the rows of its strip.  The DCP_NSTEPS steps of
// one launch are a pipeline of time levels in registers: when row j of the
// input arrives, level l finishes row j - l*RY.  A level keeps no rows: an
// arriving row is added at once to the 2*RY partial sums per column that it
// touches (DcpRow, generated), so a level's state is 2*RY values per column
// and each row costs its sums plus two lane exchanges.  Device memory is read
// once (plus the strip overlap) and written once per DCP_NSTEPS steps.
//
// Input rows reach the warp through a ring of DCP_R rows in shared memory that
// belongs to it alone, filled by asynchronous copies DCP_R - 2 rows ahead: no
// block barrier, no register and no scoreboard is held by a load in flight.
// (Rows prefetched into registers instead left each row waiting for about one
// memory latency, 0.75 us whatever the number of levels: a warp has six
// scoreboards, and the lane exchanges need them too.)
//
// Measured on a GB300 against the form that kept 2*RY + 1 rows per level and
// read them element by element (with the planner's depth and rows per item):
// 4000 x 4100 binary32, fixed ring, 50 steps 526 -> 291 us; 2047 x 2051
// binary64, periodic, 20 steps 723 (shared-memory tiles) -> 567 us; 4096
// binary32 instances of 32^2 to 512^2, 20 steps 2.84 -> 1.83 ms; the 20-step
// reverse pass of a 4096^2 binary32 chain with its loss 3.01 -> 1.69 ms; four
// steps of 10^8 binary32 elements, zero boundary, 242 -> 209 us.
//
// Work items are (array, strip, row segment); a segment streams its rows plus
// NSTEPS*RY warm-up rows above and below it.  Warps stride through the items
// (items of the largest arrays first in batched launches).  A strip writes
// DCP_W columns starting at a multiple of C, its first lane HX (the halo
// rounded up to whole vectors) columns to the left, so that rows of a 16-byte
// multiple are read and written in whole vectors; other row lengths fall back
// to the widest access that divides them.  Strips of 1-D binary64 arrays are
// as wide as their halos allow and go element by element: the FP64 pipe bounds
// them, and vectors cost a step 2 of 62 columns.
//
// Boundaries: ZERO clears the columns (CHECK strips) and rows outside the
// array at every level; FIXED_RING lets the sums of ring cells carry the
// cell's own value; PERIODIC reads rows and columns at their wrapped
// positions and computes the copies like the cells they copy.
//
// Bound: instruction issue (binary32) or the FP64 pipe (binary64).  Per level
// and row a 5-point binary32 step issues 20 arithmetic instructions and 2
// shuffles for 128 columns.
//
// The generated prefix defines DCP_T, DCP_C, DCP_RX, DCP_RY, DCP_NSTEPS,
// DCP_BC, DCP_THREADS, DCP_KNAME, DCP_BATCH, DCP_LAST, DCP_R, DCP_GUARD,
// DCP_MINB, DCP_W, DCP_HX, DCP_VEC (elements per access, 0: per instance),
// DCP_HUGE, DCP_NLOAD, DCP_NIN = max(1, DCP_NLOAD), DCP_PRO, DCP_POST (maps or reductions
// after the last step), DCP_NSTORE, DCP_NRED, DCP_NSCALAR, dcp_red_op(r) and
//   T    dcp_pro(const T (&ld)[DCP_NIN], const T* sc)     input maps on the loaded values
//   struct DcpRow<L>::run<RINGM>(a, st, out, km, rm)      arrival of row a in level L+1
//   T    dcp_epi<L>(T v)                 epilogue maps fused after step L
//   void dcp_post(const DcpStParams& p, const T* sc, long long i, T v, T* st, T* rv)
typedef DCP_T T;
typedef typename DcpFin<T>::type F;
#define DCP_ARR(n) ((n) > 0 ? (n) : 1)
#ifndef DCP_MINB
#define DCP_MINB 1   // CTAs per SM the compiler's register budget must allow
#endif

#define DCP_BC_ZERO 0
#define DCP_BC_PERIODIC 1
#define DCP_BC_FIXED_RING 2

constexpr int K = DCP_NSTEPS;
constexpr int C = DCP_C;
constexpr int RY = DCP_RY;
constexpr int NST = DCP_ARR(2 * RY);               // partial sums per column and level
constexpr int SPAN = 32 * C;                       // columns held by a warp
constexpr int HX = DCP_HX;                         // left halo, whole vectors (DCP_VEC 1: any)
constexpr int W = DCP_W;                           // columns written by a warp
static_assert(W > 0 && HX + W + K * DCP_RX <= SPAN, "strip too narrow for the number of steps");
static_assert(DCP_VEC == 1 || (W % C == 0 && HX % C == 0), "strips start on vector boundaries");
constexpr int RING = DCP_BC == DCP_BC_FIXED_RING ? RY : 0;  // ring rows

constexpr int R = DCP_R;                           // rows of a warp's ring
constexpr int D = R - 2;                           // rows requested ahead (rows go in pairs)
constexpr int ROWB = SPAN * (int)sizeof(T);        // bytes of a row
static_assert(R >= 4, "the ring holds a pair of rows, the pair before and one ahead");

typedef DcpStParamsT<T> DcpStParams;

// Sums of columns.  In rows within a strip of 2^31 columns (DCP_HUGE) those past
// 2^31 - 1, beyond the row's end, come as negative numbers below any halo's.
#if DCP_HUGE
#define DCP_PLUS(a, b) ((int)((unsigned)(a) + (unsigned)(b)))
#else
#define DCP_PLUS(a, b) (a + b)
#endif

__device__ __forceinline__ int dcp_wrap(int q, int n) {
  if ((unsigned)q < (unsigned)n) return q;
  if (DCP_HUGE && q < -(1 << 30)) return (int)((unsigned)q % (unsigned)n);
  int r = q % n;
  return r < 0 ? r + n : r;
}

// V consecutive elements as one access.
template <int V> struct DcpAcc;
template <> struct DcpAcc<1> { typedef T type; };
template <> struct DcpAcc<2> { typedef typename DcpVec2<T>::type type; };
template <> struct DcpAcc<4> { typedef uint4 type; };  // C = 4: binary32

// Asynchronous copy of V elements into the ring: `n` bytes of them from src
// (all or none), zeros for the rest.
template <int V>
__device__ __forceinline__ void dcp_copy(unsigned dst, const T* src, int n) {
  constexpr int B = V * (int)sizeof(T);
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(B), "r"(n) : "memory");
}
__device__ __forceinline__ void dcp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void dcp_wait_copies() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// One array (or instance) and the part of it a work item covers.
struct DcpItem {
  const T* in[DCP_NIN];
  int ny, nx;
  int x0;        // first written column
  int y0, y1;    // rows written
  int vec;       // batched: elements per access (C: 16-byte rows, else 2 or 1)
};

// The lane's columns in a work item.
struct DcpCols {
  int col0;
  unsigned ring;                       // bit c: the column belongs to a fixed ring
  typename DcpBits<T>::type keep[C];   // all ones inside the array, else 0
  // Copies: access i of a lane covers unit lane + 32 i of the strip (units of V
  // elements), so that a warp's copies are contiguous.
  unsigned in;                         // bit i: access i lies inside the array
  int pcol[C];                         // periodic CHECK strips: the wrapped column of access i (V = 1)
  unsigned dst;                        // shared address of the warp's ring, at the lane's vector
};

// CHECK: the strip reaches outside the array (per-column tests).  ROWS: every
// row this iteration touches lies inside the array and outside a fixed ring.
template <int L, bool CHECK, bool ROWS>
__device__ __forceinline__ void dcp_levels(T (&a)[C], T (&st)[K][NST][C], int j, const DcpItem& it,
                                           const DcpCols& cols, const T (&km)[DCP_NK]) {
  if constexpr (L < K) {
    constexpr bool RINGM = DCP_BC == DCP_BC_FIXED_RING && (CHECK || !ROWS);
    const int y = j - (L + 1) * RY;  // the row this level finishes
    unsigned rm[RY + 1];
#pragma unroll
    for (int k = 0; k <= RY; ++k) {
      rm[k] = 0u;
      if (RINGM) {
        const bool rr = !ROWS && (y + k < RY || y + k >= it.ny - RY);
        rm[k] = rr ? ~0u : cols.ring;
      }
    }
    T v[C];
    DcpRow<L>::template run<RINGM>(a, st[L], v, km, rm);
#pragma unroll
    for (int c = 0; c < C; ++c) v[c] = dcp_epi<L>(v[c]);
    if (DCP_BC == DCP_BC_ZERO) {
      // ghost zeros at every level, exact for any value an epilogue leaves
      // there (a bitwise AND, NaN included)
      if (!ROWS && (unsigned)y >= (unsigned)it.ny) {
#pragma unroll
        for (int c = 0; c < C; ++c) v[c] = (T)0;
      } else if (CHECK) {
#pragma unroll
        for (int c = 0; c < C; ++c) v[c] = dcp_keep(v[c], cols.keep[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) a[c] = v[c];
    dcp_levels<L + 1, CHECK, ROWS>(a, st, j, it, cols, km);
  }
}

template <int V>
__device__ __forceinline__ void dcp_st_row(T* p, const T (&src)[C], unsigned in) {
  typedef typename DcpAcc<V>::type A;
#pragma unroll
  for (int u = 0; u < C / V; ++u) {
    union { A a; T t[V]; } x;
#pragma unroll
    for (int v = 0; v < V; ++v) x.t[v] = src[u * V + v];
    if ((in >> (u * V)) & 1u) *reinterpret_cast<A*>(p + u * V) = x.a;
  }
}

// Copies of one row: p points at the lane's first unit, dst at the lane's
// 16-byte vector of the ring row.
template <int V, bool CHECK>
__device__ __forceinline__ void dcp_copy_row(unsigned dst, const T* p, unsigned in) {
  constexpr int B = V * (int)sizeof(T);
  dst -= (threadIdx.x & 31) * (16 - B);
#pragma unroll
  for (int i = 0; i < C / V; ++i)
    dcp_copy<V>(dst + 32 * i * B, p + 32 * i * V, !CHECK || ((in >> i) & 1u) ? B : 0);
}

// Elements per copy of the strip.
template <bool CHECK>
__device__ __forceinline__ int dcp_vec(const DcpItem& it) {
  if (DCP_BC == DCP_BC_PERIODIC && CHECK) return 1;
  return DCP_VEC > 0 ? DCP_VEC : it.vec;
}

// Requests row `row` of the array (src: its first unit of the lane, per input)
// into ring row `so`; CHECK: only the accesses of `in`.
template <bool CHECK>
__device__ __forceinline__ void dcp_request(unsigned so, const T* const (&src)[DCP_NIN], unsigned in,
                                            const DcpItem& it, const DcpCols& cols) {
#pragma unroll
  for (int l = 0; l < DCP_NLOAD; ++l) {
    const unsigned dst = cols.dst + l * (R * ROWB) + so;
    if (DCP_BC == DCP_BC_PERIODIC && CHECK) {
      // src: the row's first column
#pragma unroll
      for (int i = 0; i < C; ++i)
        dcp_copy<1>(dst - (threadIdx.x & 31) * (16 - (int)sizeof(T)) + 32 * i * (int)sizeof(T),
                    src[l] + cols.pcol[i], (int)sizeof(T));
    } else {
      const int vec = dcp_vec<CHECK>(it);
      if (vec == C) dcp_copy_row<C, CHECK>(dst, src[l], in);
      else if (C > 2 && vec == 2) dcp_copy_row<2, CHECK>(dst, src[l], in);
      else dcp_copy_row<1, CHECK>(dst, src[l], in);
    }
  }
  dcp_commit();
}

// The lane's first unit of row `row` in every input (periodic CHECK strips:
// the row's first column).
template <bool CHECK>
__device__ __forceinline__ void dcp_src(const T* (&src)[DCP_NIN], int row, const DcpItem& it) {
  const long long at = (long long)row * it.nx +
                       (DCP_BC == DCP_BC_PERIODIC && CHECK
                            ? 0 : it.x0 - HX + (int)(threadIdx.x & 31) * dcp_vec<CHECK>(it));
#pragma unroll
  for (int l = 0; l < DCP_NLOAD; ++l) src[l] = it.in[l] + at;
}

// Requests input row j with its boundary tests (zeros outside the array).  An
// item of a 1-D array is one row: the rows after it are only counted.
template <bool CHECK>
__device__ __forceinline__ void dcp_request_checked(unsigned so, int j, const DcpItem& it,
                                                    const DcpCols& cols) {
  if (RY == 0 && j >= it.y1) {
    dcp_commit();
    return;
  }
  const bool inside = (unsigned)j < (unsigned)it.ny;
  const T* src[DCP_NIN];
  dcp_src<CHECK>(src, DCP_BC == DCP_BC_PERIODIC ? dcp_wrap(j, it.ny) : (inside ? j : 0), it);
  if (DCP_BC == DCP_BC_PERIODIC) dcp_request<CHECK>(so, src, cols.in, it, cols);
  else dcp_request<true>(so, src, inside ? cols.in : 0u, it, cols);
}

constexpr unsigned RMASK = R * ROWB - 1;  // ring offsets wrap by a mask
static_assert((R & (R - 1)) == 0, "power-of-two ring");

union DcpRaw { uint4 v; T t[C]; };

// The lane's vector of ring row `so`, per input.
__device__ __forceinline__ void dcp_load(DcpRaw (&x)[DCP_NIN], unsigned so, const DcpCols& cols) {
  if (DCP_NLOAD == 0) x[0].v = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int l = 0; l < DCP_NLOAD; ++l)
    asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(x[l].v.x), "=r"(x[l].v.y), "=r"(x[l].v.z), "=r"(x[l].v.w)
                 : "r"(cols.dst + l * (R * ROWB) + so)
                 : "memory");
}

// Input row j (its loaded vectors x) through every level; `a` ends as row
// j - K*RY after the last.
template <bool CHECK, bool ROWS, class Pro>
__device__ __forceinline__ void dcp_row(T (&a)[C], T (&st)[K][NST][C], const DcpRaw (&x)[DCP_NIN], int j,
                                        const DcpItem& it, const DcpCols& cols,
                                        const T (&km)[DCP_NK], Pro& pro, DcpGuard& guard) {
#pragma unroll
  for (int c = 0; c < C; ++c) {
    T ld[DCP_NIN];
#pragma unroll
    for (int l = 0; l < DCP_NIN; ++l) ld[l] = x[l].t[c];
    a[c] = pro(ld);
  }
  if (DCP_PRO && DCP_BC != DCP_BC_PERIODIC) {
    // the maps of the zeros read outside the array need not be 0
    if (!ROWS && (unsigned)j >= (unsigned)it.ny) {
#pragma unroll
      for (int c = 0; c < C; ++c) a[c] = (T)0;
    } else if (CHECK) {
#pragma unroll
      for (int c = 0; c < C; ++c) a[c] = dcp_keep(a[c], cols.keep[c]);
    }
  }
  if (DCP_GUARD) {
#pragma unroll
    for (int c = 0; c < C; ++c) guard.see(a[c]);
  }
  dcp_levels<0, CHECK, ROWS>(a, st, j, it, cols, km);
}

template <bool CHECK, class Pro, class Output>
__device__ __forceinline__ void dcp_stream_impl(const DcpItem& it, Pro& pro, Output& output,
                                                DcpGuard& guard, const T (&km)[DCP_NK]) {
  extern __shared__ __align__(16) unsigned char dcp_smem[];
  const int lane = threadIdx.x & 31;
  DcpCols cols;
  const int col0 = DCP_PLUS(it.x0 - HX, lane * C);
  cols.dst = (unsigned)__cvta_generic_to_shared(dcp_smem) +
             (threadIdx.x >> 5) * (DCP_NIN * R * ROWB) + lane * 16;
  cols.ring = cols.in = 0u;
  const int vec = dcp_vec<CHECK>(it);
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int col = DCP_PLUS(col0, c);
    if (CHECK) cols.ring |= col < DCP_RX || col >= it.nx - DCP_RX ? 1u << c : 0u;
    cols.keep[c] = (unsigned)col < (unsigned)it.nx ? ~(typename DcpBits<T>::type)0 : 0;
    const int u = DCP_PLUS(it.x0 - HX, (lane + 32 * c) * vec);  // first column of access c
    cols.in |= (unsigned)u < (unsigned)it.nx ? 1u << c : 0u;
    if (CHECK && DCP_BC == DCP_BC_PERIODIC) cols.pcol[c] = dcp_wrap(u, it.nx);
  }
  // Rows before the first streamed row count as zeros: exact ghosts above the
  // array; inside the array they only feed warm-up rows that are never written.
  T st[K][NST][C];
#pragma unroll
  for (int l = 0; l < K; ++l)
#pragma unroll
    for (int d = 0; d < NST; ++d)
#pragma unroll
      for (int c = 0; c < C; ++c) st[l][d][c] = (T)0;
  int j = it.y0 - K * RY;
  const int jend = it.y1 + K * RY;   // rows j >= jout finish a written row
  const int jout = it.y0 + K * RY;
  unsigned so = 0;                   // ring offset of row j
  __syncwarp();  // the previous item's rows have been read
  for (int r = 0; r < D; ++r) dcp_request_checked<CHECK>(r * ROWB, j + r, it, cols);
  // Rows [f0, f1] run without row tests: every row such an iteration touches
  // -- level rows from j - K*RY, the requested row j + D -- lies inside the
  // array and outside a fixed ring (periodic: the requested row).  They go in
  // pairs (j, j + 1), j < f1.
  const int f0 = DCP_BC == DCP_BC_PERIODIC ? -D : K * RY + RING;
  const int f1 = min(jend - 1, it.ny - (DCP_BC == DCP_BC_PERIODIC ? 0 : RING) - 1 - D);
  T a[C];
  while (j < jend) {
    if (j >= f0 && j < f1) {
      const T* src[DCP_NIN];
      dcp_src<CHECK>(src, j + D, it);
      long long gi = (long long)(j - K * RY) * it.nx + col0;  // the lane's first element of the finished row
#pragma unroll 1
      do {
        // two rows per wait: their levels interleave, and the partial sums
        // alternate registers
        dcp_wait_copies<D - 2>();  // this lane's copies of rows j and j + 1 have landed
        __syncwarp();              // every lane's have, and the pair before has been read
        DcpRaw x0[DCP_NIN], x1[DCP_NIN];
        dcp_load(x0, so, cols);
        dcp_load(x1, (so + ROWB) & RMASK, cols);
#pragma unroll
        for (int h = 2; h >= 1; --h) {
          dcp_request<CHECK>((so - h * ROWB) & RMASK, src, cols.in, it, cols);
#pragma unroll
          for (int l = 0; l < DCP_NLOAD; ++l) src[l] += it.nx;
        }
        so = (so + 2 * ROWB) & RMASK;
        dcp_row<CHECK, true>(a, st, x0, j, it, cols, km, pro, guard);
        if (j >= jout) output(gi, a);
        gi += it.nx;
        dcp_row<CHECK, true>(a, st, x1, j + 1, it, cols, km, pro, guard);
        if (j + 1 >= jout) output(gi, a);
        gi += it.nx;
        j += 2;
      } while (j < f1);
    }
    if (j < jend) {
      dcp_wait_copies<D - 1>();
      __syncwarp();
      DcpRaw x[DCP_NIN];
      dcp_load(x, so, cols);
      dcp_request_checked<CHECK>((so - 2 * ROWB) & RMASK, j + D, it, cols);
      dcp_row<CHECK, false>(a, st, x, j, it, cols, km, pro, guard);
      so = (so + ROWB) & RMASK;
      if (j >= jout) output((long long)(j - K * RY) * it.nx + col0, a);
      ++j;
    }
  }
  dcp_wait_copies<0>();
}

// Strips whose columns all lie inside the array (outside a fixed ring) take
// the path without per-column boundary tests.
// With DCP_GUARD every row the stream reads enters the magnitude guard.
template <class Pro, class Output>
__device__ __forceinline__ void dcp_stream(const DcpItem& it, Pro&& pro, DcpGuard& guard,
                                           const T (&km)[DCP_NK], Output&& output) {
  const int lo = DCP_BC == DCP_BC_FIXED_RING ? DCP_RX : 0;
  const int first = it.x0 - HX;
  if (first >= lo && (DCP_HUGE ? first <= it.nx - lo - SPAN : first + SPAN <= it.nx - lo)) dcp_stream_impl<false>(it, pro, output, guard, km);
  else dcp_stream_impl<true>(it, pro, output, guard, km);
}

// Bit c: the lane's column c is written by the strip starting at x0.
__device__ __forceinline__ unsigned dcp_written(int x0, int nx) {
  unsigned m = 0u;
#if DCP_HUGE
  const int at = (int)(threadIdx.x & 31) * C - HX;  // the lane's first column, from x0
#pragma unroll
  for (int c = 0; c < C; ++c) m |= at + c >= 0 && at + c < W && at + c < nx - x0 ? 1u << c : 0u;
#else
  const int col0 = x0 - HX + (threadIdx.x & 31) * C;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int col = col0 + c;
    m |= col >= x0 && col < x0 + W && col < nx ? 1u << c : 0u;
  }
#endif
  return m;
}

__device__ __forceinline__ void dcp_write_row(T* p, const T (&v)[C], unsigned m, int run_vec) {
  const int vec = DCP_VEC > 0 ? DCP_VEC : run_vec;
  if (vec == C) dcp_st_row<C>(p, v, m);
  else if (C > 2 && vec == 2) dcp_st_row<2>(p, v, m);
  else dcp_st_row<1>(p, v, m);
}

#if !defined(DCP_PRO) || !defined(DCP_POST) || !defined(DCP_W)
#error "incomplete generated prefix"
#endif

#if !DCP_BATCH
// Single array: items = strips x row segments of p.seg rows; the host launches
// the variant whose DCP_VEC suits every buffer and the row length.
extern "C" __global__ void __launch_bounds__(DCP_THREADS, DCP_MINB) DCP_KNAME(const DcpStParams p) {
  T sc[DCP_ARR(DCP_NSCALAR)];
#pragma unroll
  for (int i = 0; i < DCP_NSCALAR; ++i) sc[i] = p.sc[i][0];
  T acc[DCP_ARR(DCP_NRED)];
#pragma unroll
  for (int r = 0; r < DCP_NRED; ++r) acc[r] = dcp_red_init<T>(dcp_red_op(r));
  const int ny = p.ny, nx = p.nx;
  const int strips = DCP_HUGE ? (nx - 1) / W + 1 : (nx + W - 1) / W;
  const int SEG = p.seg > 0 ? p.seg : ny;
  const int segs = (ny + SEG - 1) / SEG;
  const int items = strips * segs;
  const int warp = (blockIdx.x * DCP_THREADS + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * DCP_THREADS) >> 5;
  DcpGuard guard;
  T km[DCP_NK];
  dcp_load_multipliers(km, dcp_km);
  for (int w = warp; w < items; w += nwarps) {
    const int sg = w / strips, st = w - sg * strips;
    DcpItem it;
#pragma unroll
    for (int l = 0; l < DCP_NIN; ++l) it.in[l] = p.ld[l];
    it.ny = ny;
    it.nx = nx;
    it.x0 = st * W;
    it.y0 = sg * SEG;
    it.y1 = min(ny, it.y0 + SEG);
    it.vec = 0;
    const unsigned wm = dcp_written(it.x0, nx);
    dcp_stream(
        it, [&](const T (&ld)[DCP_NIN]) { return dcp_pro(ld, sc); }, guard, km,
        [&](long long gi, const T (&v)[C]) {
#if DCP_POST
          T sv[DCP_ARR(DCP_NSTORE)][C];
#pragma unroll
          for (int c = 0; c < C; ++c) {
            if (!((wm >> c) & 1u)) continue;
            T stv[DCP_ARR(DCP_NSTORE)], rv[DCP_ARR(DCP_NRED)];
            dcp_post(p, sc, gi + c, v[c], stv, rv);
#pragma unroll
            for (int s = 0; s < DCP_NSTORE; ++s) sv[s][c] = stv[s];
#pragma unroll
            for (int r = 0; r < DCP_NRED; ++r)
              acc[r] = dcp_red_comb(dcp_red_op(r), acc[r], dcp_red_lift(dcp_red_op(r), rv[r]));
          }
#pragma unroll
          for (int s = 0; s < DCP_NSTORE; ++s) dcp_write_row(p.st[s] + gi, sv[s], wm, 0);
#else
          dcp_write_row(p.st[0] + gi, v, wm, 0);
#endif
        });
  }
#if DCP_LAST && DCP_NRED > 0
  dcp_reduce_epilogue<T, DCP_NRED, DCP_THREADS>(acc, p.red_out, p.partials, p.ticket);
#endif
#if DCP_GUARD
  guard.flush(p.guard);
#endif
}
#else
// Batched form: items are (instance, strip, row segment); instances are
// ordered largest first by the host; the item of warp w is found by binary
// search over the instances' first item numbers.
struct DcpInst {
  const T* in;
  T* out;
  int ny, nx, tiles_x, tile0;  // tiles_x = strips of the instance, tile0 = its first item
};
struct DcpBatchParams {
  const DcpInst* inst;
  int ninst;
  int total_tiles;
  int seg;   // rows per work item
  int pad_;
  unsigned long long* guard;  // first launch of a deferred run: largest |input| seen
};

extern "C" __global__ void __launch_bounds__(DCP_THREADS, DCP_MINB) DCP_KNAME(const DcpBatchParams p) {
  const int warp = (blockIdx.x * DCP_THREADS + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * DCP_THREADS) >> 5;
  DcpGuard guard;
  T km[DCP_NK];
  dcp_load_multipliers(km, dcp_km);
  for (int w = warp; w < p.total_tiles; w += nwarps) {
    int lo = 0, hi = p.ninst - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (p.inst[mid].tile0 <= w) lo = mid;
      else hi = mid - 1;
    }
    const DcpInst I = p.inst[lo];
    const int t = w - I.tile0;
    const int sg = t / I.tiles_x, st = t - sg * I.tiles_x;
    DcpItem it;
    it.in[0] = I.in;
    it.ny = I.ny;
    it.nx = I.nx;
    it.x0 = st * W;
    it.y0 = sg * p.seg;
    it.y1 = min(I.ny, it.y0 + p.seg);
    // the widest access that suits both buffers and the row length
    const unsigned long long mis = reinterpret_cast<unsigned long long>(I.in) |
                                   reinterpret_cast<unsigned long long>(I.out) |
                                   (unsigned long long)I.nx * sizeof(T);
    it.vec = (mis & 15) == 0 ? C : (C > 2 && (mis & 7) == 0 ? 2 : 1);
    T* out = I.out;
    const int vec = it.vec;
    const unsigned wm = dcp_written(it.x0, I.nx);
    dcp_stream(
        it, [&](const T (&ld)[DCP_NIN]) { return ld[0]; }, guard, km,
        [&](long long gi, const T (&v)[C]) { dcp_write_row(out + gi, v, wm, vec); });
  }
#if DCP_GUARD
  guard.flush(p.guard);
#endif
}
#endif
