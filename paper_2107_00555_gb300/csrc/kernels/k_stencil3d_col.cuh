// k_stencil3d_col.cuh -- warp-streamed 3-D star stencil (radius 1), one or two
// steps per launch.
//
// A warp owns LX*C columns along x (C per lane, one 16-byte vector) times
// 32/LX blocks of DCP_CY rows along y and streams through z.  Planes of its block (with K rows
// and one vector of columns around it) reach it through a ring of DCP_R planes
// in shared memory that belongs to it alone, filled by asynchronous copies:
// warps share nothing and there is no block barrier.  A level keeps the
// previous plane and one partial sum per cell in registers: the arrival of
// plane j finishes plane j - 1.  With DCP_NSTEPS = 2 the finished plane of
// the first level, on one more row above and below, feeds the second.
//
// Sums.  Listed order (binary32): the in-plane points, then the point below,
// then the point above, one multiply and fused multiply-adds.  Shared pairs
// (binary64, DCP_PAIRS: a run on its deferred weight whose four points at
// y +- 1 and z +- 1 have ratio 1): D(y, z) = u(y - 1, z) + u(y, z - 1) is also
// the remaining pair of the cell at (y - 1, z - 1), so a cell takes
// (CY + 1) / CY pair sums instead of two: 5.125 FP64 operations instead of 6
// (CY = 8).
//
// Bound: the FP64 pipe (binary64); device memory, then shared-memory and
// instruction issue (binary32).  Measured on a GB300 per step against the
// planes in shared memory (k_stencil3d.cuh): 512^3 binary64 periodic on a
// deferred weight 1.40 -> 1.21 ms (0.97 of the FP64 pipe's rate for 5.125
// operations); binary32, zero boundary, 512^3 248 -> 125 us, 300 x 333 x 381
// (rows read element by element) 72 -> 57 us.
//
// The generated prefix defines DCP_T, DCP_C, DCP_CY, DCP_LX, DCP_NSTEPS, DCP_R, DCP_W,
// DCP_VEC (elements per access), DCP_PAIRS, DCP_BC, DCP_THREADS, DCP_KNAME,
// DCP_LAST, DCP_POST, DCP_GUARD, DCP_MINB, DCP_NSTORE, DCP_NRED, DCP_NSCALAR,
// dcp_red_op(r) and per step S
//   pairs (column I of the lane):
//           T dcp_d<S, I>(up, before, km)           the pair sum D
//           T dcp_in<S, I>(d, c, l, r, km)          D + the points of the row
//           T dcp_fin<S, I>(acc, d, km)             + the other pair
//   listed: T dcp_in<S>(c, l, r, up, dn, before)    all but the point above
//           T dcp_fin<S>(acc, c)                    + the point above
//   T dcp_epi<S>(T v), dcp_post(...) as in the other stencil skeletons
typedef DCP_T T;
typedef typename DcpFin<T>::type F;
#define DCP_ARR(n) ((n) > 0 ? (n) : 1)

#define DCP_BC_ZERO 0
#define DCP_BC_PERIODIC 1
#define DCP_BC_FIXED_RING 2

constexpr int K = DCP_NSTEPS;
constexpr int C = DCP_C;
constexpr int CY = DCP_CY;
constexpr int LX = DCP_LX;                     // lanes along x
constexpr int LY = 32 / LX;                    // blocks of CY rows a warp covers
constexpr int SPAN = LX * C;
constexpr int HX = K > 1 ? C : 0;              // the second level loses its edge lanes
constexpr int W = DCP_W;                       // columns written
static_assert(W == SPAN - 2 * HX && (K == 1 || LX == 32), "columns written");
constexpr int ROWE = SPAN + 2 * C;             // ring row: one vector on either side
constexpr int ROWS = LY * CY + 2 * K;          // ring rows of a plane: y0 - K ..
constexpr int PLANEB = ROWS * ROWE * (int)sizeof(T);
constexpr int R = DCP_R;                       // planes of the ring
constexpr int D = R - 1;                       // planes requested ahead
constexpr int V = DCP_VEC;
constexpr int NM = C / V;                      // copies of a row per lane
constexpr int NG = ROWS / LY;                  // groups of LY rows
constexpr int EPR = 2 * C / V;                 // copies of a row's edge vectors
constexpr int NE = (ROWS * EPR + 31) / 32;     // edge copies per lane and plane
static_assert(ROWS % LY == 0, "whole row groups");

typedef DcpStParamsT<T> DcpStParams;

template <int N> struct DcpAcc;
template <> struct DcpAcc<1> { typedef T type; };
template <> struct DcpAcc<2> { typedef typename DcpVec2<T>::type type; };
template <> struct DcpAcc<4> { typedef uint4 type; };  // C = 4: binary32

__device__ __forceinline__ int dcp_wrap(int q, int n) {
  if ((unsigned)q < (unsigned)n) return q;
  int r = q % n;
  return r < 0 ? r + n : r;
}

template <int N>
__device__ __forceinline__ void dcp_copy(unsigned dst, const T* src, int n) {
  constexpr int B = N * (int)sizeof(T);
  if constexpr (B == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(B), "r"(n) : "memory");
}

struct DcpItem {
  const T* in;
  int nz, ny, nx;
  int x0, y0, z0, z1;
  unsigned ring;      // shared address of the warp's ring
};

// What the lane copies of every plane, fixed for a work item: copy i of row
// group g covers unit lx + LX i of row g LY + ly, the edge vectors of all rows
// are dealt to the lanes in turn.  Rows and columns outside the array are
// filled with zeros (periodic: taken at their wrapped positions).
template <bool CHECK> struct DcpLane {
  unsigned in;                         // bit i: main copy i lies inside the array
  unsigned rows;                       // bit g: the lane's row of group g does
  bool wrapped;                        // periodic: the block reaches over an edge along y
  int col[NM];                         // periodic CHECK strips: wrapped columns
  int eoff[NE];                        // edge copies: offset in the plane (-1: zeros)
  unsigned ringc;                      // bit c: column c belongs to a fixed ring
  typename DcpBits<T>::type keep[C];
  __device__ __forceinline__ DcpLane(const DcpItem& it) {
    const int lane = threadIdx.x & 31, lx = lane % LX, ly = lane / LX;
    in = ringc = rows = 0u;
    wrapped = DCP_BC == DCP_BC_PERIODIC && (it.y0 - K < 0 || it.y0 - K + ROWS > it.ny);
#pragma unroll
    for (int i = 0; i < NM; ++i) {
      const int x = it.x0 - HX + (lx + LX * i) * V;
      if ((unsigned)x < (unsigned)it.nx || DCP_BC == DCP_BC_PERIODIC) in |= 1u << i;
      col[i] = dcp_wrap(x, it.nx);
    }
#pragma unroll
    for (int g = 0; g < NG; ++g)
      if ((unsigned)(it.y0 - K + g * LY + ly) < (unsigned)it.ny || DCP_BC == DCP_BC_PERIODIC) rows |= 1u << g;
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int e = lane + 32 * i, r = e / EPR, u = e - r * EPR;
      int y = it.y0 - K + r, x = it.x0 - HX + (u < C / V ? u * V - C : SPAN + u * V - C);
      if (DCP_BC == DCP_BC_PERIODIC) {
        y = dcp_wrap(y, it.ny);
        x = dcp_wrap(x, it.nx);
      }
      const bool ok = e < ROWS * EPR && (unsigned)y < (unsigned)it.ny && (unsigned)x < (unsigned)it.nx;
      eoff[i] = ok ? y * it.nx + x : -1;
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int x = it.x0 - HX + lx * C + c;
      keep[c] = (unsigned)x < (unsigned)it.nx ? ~(typename DcpBits<T>::type)0 : 0;
      if (CHECK && (x < 1 || x >= it.nx - 1)) ringc |= 1u << c;
    }
  }
};

// Requests plane j into ring slot `slot` (zeros outside the array).
template <bool CHECK>
__device__ __forceinline__ void dcp_request(int slot, int j, const DcpItem& it,
                                            const DcpLane<CHECK>& ln) {
  constexpr int B = V * (int)sizeof(T);
  const int lane = threadIdx.x & 31, lx = lane % LX, ly = lane / LX;
  if (j < it.z1 + K) {  // (else past the last plane the item reads)
    const bool plane_ok = DCP_BC == DCP_BC_PERIODIC || (unsigned)j < (unsigned)it.nz;
    const int z = DCP_BC == DCP_BC_PERIODIC ? dcp_wrap(j, it.nz) : (plane_ok ? j : 0);
    const T* plane = it.in + (long long)z * it.ny * it.nx;
    const unsigned ring = it.ring + slot * PLANEB;
    const unsigned rows = plane_ok ? ln.rows : 0u;
    const unsigned dst = ring + (ly * ROWE + C + lx * V) * (int)sizeof(T);
    if (DCP_BC == DCP_BC_PERIODIC && (CHECK || ln.wrapped)) {
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        const T* p = plane + (long long)dcp_wrap(it.y0 - K + g * LY + ly, it.ny) * it.nx;
#pragma unroll
        for (int i = 0; i < NM; ++i)
          dcp_copy<V>(dst + (g * LY * ROWE + LX * i * V) * (int)sizeof(T), p + ln.col[i], B);
      }
    } else {
      const T* p = plane + (long long)(it.y0 - K + ly) * it.nx + (it.x0 - HX + lx * V);
      const long long step = (long long)LY * it.nx;
      constexpr unsigned ALL = NG < 32 ? (1u << NG) - 1u : ~0u;
      if (!CHECK && __all_sync(0xffffffffu, rows == ALL)) {
#pragma unroll
        for (int g = 0; g < NG; ++g, p += step)
#pragma unroll
          for (int i = 0; i < NM; ++i)
            dcp_copy<V>(dst + (g * LY * ROWE + LX * i * V) * (int)sizeof(T), p + LX * i * V, B);
      } else {
        int n[NM];
#pragma unroll
        for (int i = 0; i < NM; ++i) n[i] = (ln.in >> i) & 1u ? B : 0;
#pragma unroll
        for (int g = 0; g < NG; ++g, p += step)
#pragma unroll
          for (int i = 0; i < NM; ++i)
            dcp_copy<V>(dst + (g * LY * ROWE + LX * i * V) * (int)sizeof(T), p + LX * i * V,
                        (rows >> g) & 1u ? n[i] : 0);
      }
    }
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      const int e = lane + 32 * i, r = e / EPR, u = e - r * EPR;
      if (ROWS * EPR % 32 != 0 && e >= ROWS * EPR) break;
      const bool ok = plane_ok && ln.eoff[i] >= 0;
      dcp_copy<V>(ring + (r * ROWE + (u < C / V ? u * V : SPAN + u * V)) * (int)sizeof(T),
                  plane + (ok ? ln.eoff[i] : 0), ok ? B : 0);
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

struct DcpRow {
  T v[C];
};

__device__ __forceinline__ void dcp_ld_row(DcpRow& a, unsigned row) {
  union { uint4 q; T t[C]; } x;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(x.q.x), "=r"(x.q.y), "=r"(x.q.z), "=r"(x.q.w)
               : "r"(row + (C + (threadIdx.x & (LX - 1)) * C) * (int)sizeof(T)) : "memory");
#pragma unroll
  for (int c = 0; c < C; ++c) a.v[c] = x.t[c];
}

// The columns left and right of the lane's.
__device__ __forceinline__ void dcp_ld_sides(T& l, T& r, unsigned row) {
  const unsigned p = row + (C + (threadIdx.x & (LX - 1)) * C) * (int)sizeof(T);
  if constexpr (sizeof(T) == 8) {
    unsigned long long a, b;
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(a) : "r"(p - 8) : "memory");
    asm volatile("ld.shared.u64 %0, [%1];" : "=l"(b) : "r"(p + C * 8) : "memory");
    l = __longlong_as_double((long long)a);
    r = __longlong_as_double((long long)b);
  } else {
    unsigned a, b;
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(a) : "r"(p - 4) : "memory");
    asm volatile("ld.shared.u32 %0, [%1];" : "=r"(b) : "r"(p + C * 4) : "memory");
    l = __uint_as_float(a);
    r = __uint_as_float(b);
  }
}

// Per level: the previous plane and the partial sums of the rows it finishes
// (N rows; `before` of the pair form holds one row more).
template <int N> struct DcpState {
  T before[N + 1][C];
  T acc[N][C];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int r = 0; r <= N; ++r)
#pragma unroll
      for (int c = 0; c < C; ++c) before[r][c] = (T)0;
#pragma unroll
    for (int r = 0; r < N; ++r)
#pragma unroll
      for (int c = 0; c < C; ++c) acc[r][c] = (T)0;
  }
};

#if DCP_PAIRS
// The generated sums of the lane's columns (one instance per column: each
// keeps multiplier registers of its own, see dcp_load_multipliers).
template <int S, int I>
__device__ __forceinline__ void dcp_pair(T (&d)[C], const T (&up)[C], const T (&before)[C], const T (&km)[DCP_NK]) {
  if constexpr (I < C) {
    d[I] = dcp_d<S, I>(up[I], before[I], km);
    dcp_pair<S, I + 1>(d, up, before, km);
  }
}
template <int S, int I>
__device__ __forceinline__ void dcp_inner(T (&a)[C], const T (&d)[C], const T (&c)[C], T l, T r, const T (&km)[DCP_NK]) {
  if constexpr (I < C) {
    a[I] = dcp_in<S, I>(d[I], c[I], I > 0 ? c[I > 0 ? I - 1 : 0] : l, I + 1 < C ? c[I + 1 < C ? I + 1 : 0] : r, km);
    dcp_inner<S, I + 1>(a, d, c, l, r, km);
  }
}
template <int S, int I>
__device__ __forceinline__ void dcp_finish(T (&o)[C], const T (&acc)[C], const T (&d)[C], const T (&km)[DCP_NK]) {
  if constexpr (I < C) {
    o[I] = dcp_fin<S, I>(acc[I], d[I], km);
    dcp_finish<S, I + 1>(o, acc, d, km);
  }
}
#endif

// Plane j arrives at step S, whose rows y, y + 1, .. the level finishes on
// plane j - 1.  get(r, row) gives row r = -1 .. N of the arriving plane,
// sides(r, row, l, rt) the columns beside the lane's of row r = 0 .. N - 1.
// LAST (pair form): the plane's own sums are not needed.
template <int S, int N, bool LAST, class Get, class Sides>
__device__ __forceinline__ void dcp_arrive(DcpState<N>& st, T (&out)[N][C], int j, int y,
                                           const DcpItem& it, unsigned ringc,
                                           const T (&km)[DCP_NK], Get&& get, Sides&& sides) {
  // fixed ring: a cell's sum is its own value (set on its plane's arrival,
  // kept when the next plane finishes it); deferred runs, the pair form, have none
  constexpr bool RINGM = DCP_BC == DCP_BC_FIXED_RING;
  static_assert(!(DCP_PAIRS && RINGM), "a deferred run has no fixed ring");
  const bool rz0 = RINGM && (j < 1 || j >= it.nz - 1), rz1 = RINGM && (j - 1 < 1 || j - 1 >= it.nz - 1);
  auto ring = [&](int r, bool rz) -> unsigned {
    return rz || y + r < 1 || y + r >= it.ny - 1 ? ~0u : ringc;
  };
  DcpRow up, cur, dn;
  T pend[C];  // pair form: a row's new sum, until its old one is finished
  (void)pend;
  get(-1, up);
  get(0, cur);
#pragma unroll
  for (int r = 0; r < N + DCP_PAIRS; ++r) {
    if (r < N) get(r + 1, dn);
#if DCP_PAIRS
    T d[C];
    dcp_pair<S, 0>(d, up.v, st.before[r], km);
    if (r > 0) {
      dcp_finish<S, 0>(out[r - 1], st.acc[r - 1], d, km);
#pragma unroll
      for (int c = 0; c < C; ++c)
        if (!LAST) st.acc[r - 1][c] = pend[c];
    }
    if (r < N && !LAST) {
      T l, rt;
      sides(r, cur, l, rt);
      dcp_inner<S, 0>(pend, d, cur.v, l, rt, km);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) st.before[r][c] = cur.v[c];
#else
    T l, rt;
    sides(r, cur, l, rt);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      out[r][c] = dcp_fin<S>(st.acc[r][c], cur.v[c]);
      if (RINGM && ((ring(r, rz1) >> c) & 1u)) out[r][c] = st.acc[r][c];
      st.acc[r][c] = dcp_in<S>(cur.v[c], c > 0 ? cur.v[c - 1] : l, c + 1 < C ? cur.v[c + 1] : rt,
                               up.v[c], dn.v[c], st.before[r][c]);
      if (RINGM && ((ring(r, rz0) >> c) & 1u)) st.acc[r][c] = cur.v[c];
      st.before[r][c] = cur.v[c];
    }
#endif
    up = cur;
    cur = dn;
  }
#pragma unroll
  for (int r = 0; r < N; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c) out[r][c] = dcp_epi<S>(out[r][c]);
}

// The first plane of the pair form: nothing to finish, and its own sums are
// not needed (binary32 levels just run on it: less code, fewer registers).
template <int N, class Get>
__device__ __forceinline__ void dcp_first(DcpState<N>& st, Get&& get) {
#pragma unroll
  for (int r = 0; r < N + DCP_PAIRS; ++r) {
    DcpRow a;
    get(r, a);
#pragma unroll
    for (int c = 0; c < C; ++c) st.before[r][c] = a.v[c];
  }
}

// Plane j (ring address pl) through the levels.
template <bool CHECK, bool LAST, class Output>
__device__ __forceinline__ void dcp_plane(DcpState<CY + 2 * (K - 1)>& s1, DcpState<CY>& s2, int j,
                                          unsigned pl, const DcpItem& it, const DcpLane<CHECK>& ln,
                                          Output& output, DcpGuard& guard, const T (&km)[DCP_NK]) {
  constexpr int N1 = CY + 2 * (K - 1);  // rows the first level finishes
  const int ly = (threadIdx.x & 31) / LX;
  auto get = [&](int r, DcpRow& a) {
    dcp_ld_row(a, pl + (ly * CY + r + 1) * ROWE * (int)sizeof(T));
    if (DCP_GUARD) {
#pragma unroll
      for (int c = 0; c < C; ++c) guard.see(a.v[c]);
    }
  };
  if (DCP_PAIRS && j == it.z0 - K) {
    dcp_first(s1, get);
    return;
  }
  T v[N1][C];
  dcp_arrive<0, N1, LAST>(s1, v, j, it.y0 - (K - 1) + ly * CY, it, ln.ringc, km, get,
                          [&](int r, const DcpRow&, T& l, T& rt) {
                            dcp_ld_sides(l, rt, pl + (ly * CY + r + 1) * ROWE * (int)sizeof(T));
                          });
  if constexpr (K > 1) {
    if (DCP_BC == DCP_BC_ZERO) {
      // ghost zeros between the steps
      const bool pin = (unsigned)(j - 1) < (unsigned)it.nz;
#pragma unroll
      for (int r = 0; r < N1; ++r) {
        const bool rin = pin && (unsigned)(it.y0 - 1 + r) < (unsigned)it.ny;
        if (!rin) {
#pragma unroll
          for (int c = 0; c < C; ++c) v[r][c] = (T)0;
        } else if (CHECK) {
#pragma unroll
          for (int c = 0; c < C; ++c) v[r][c] = dcp_keep(v[r][c], ln.keep[c]);
        }
      }
    }
    auto get2 = [&](int r, DcpRow& a) {
#pragma unroll
      for (int c = 0; c < C; ++c) a.v[c] = v[r + 1][c];
    };
    T w[CY][C];
    dcp_arrive<1, CY, LAST>(s2, w, j - 1, it.y0, it, ln.ringc, km, get2,
                            [&](int, const DcpRow& a, T& l, T& rt) {
                              l = __shfl_up_sync(0xffffffffu, a.v[C - 1], 1);
                              rt = __shfl_down_sync(0xffffffffu, a.v[0], 1);
                            });
    if (j >= it.z0 + K) output(j - K, w);
  } else {
    if (j >= it.z0 + K) output(j - K, v);
  }
}

template <bool CHECK, class Output>
__device__ __forceinline__ void dcp_column(const DcpItem& it, Output& output, DcpGuard& guard,
                                           const T (&km)[DCP_NK]) {
  const DcpLane<CHECK> ln(it);
  DcpState<CY + 2 * (K - 1)> s1;
  s1.clear();
  DcpState<CY> s2;
  if (K > 1) s2.clear();
  __syncwarp();  // the previous item's planes have been read
  int slot = 0;
  for (int r = 0; r < D; ++r) dcp_request<CHECK>(r, it.z0 - K + r, it, ln);
  const int jend = it.z1 + K;
#pragma unroll 1
  for (int j = it.z0 - K; j < jend; ++j) {
    asm volatile("cp.async.wait_group %0;" ::"n"(D - 1) : "memory");
    __syncwarp();  // every lane's copies of plane j have landed, plane j - 1 has been read
    dcp_request<CHECK>(slot == 0 ? R - 1 : slot - 1, j + D, it, ln);
    const unsigned pl = it.ring + slot * PLANEB;
    slot = slot + 1 == R ? 0 : slot + 1;
    if (DCP_PAIRS && j == jend - 1) dcp_plane<CHECK, true>(s1, s2, j, pl, it, ln, output, guard, km);
    else dcp_plane<CHECK, false>(s1, s2, j, pl, it, ln, output, guard, km);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// Items: strips of W columns x blocks of CY rows x segments of p.seg planes.
extern "C" __global__ void __launch_bounds__(DCP_THREADS, DCP_MINB) DCP_KNAME(const DcpStParams p) {
  extern __shared__ __align__(16) unsigned char dcp_smem[];
  T sc[DCP_ARR(DCP_NSCALAR)];
#pragma unroll
  for (int i = 0; i < DCP_NSCALAR; ++i) sc[i] = p.sc[i][0];
  T acc[DCP_ARR(DCP_NRED)];
#pragma unroll
  for (int r = 0; r < DCP_NRED; ++r) acc[r] = dcp_red_init<T>(dcp_red_op(r));
  const int strips = (p.nx + W - 1) / W, blocks = (p.ny + LY * CY - 1) / (LY * CY);
  const int segs = (p.nz + p.seg - 1) / p.seg;
  const long long items = (long long)strips * blocks * segs;
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * DCP_THREADS + threadIdx.x) >> 5;
  const int nwarps = (gridDim.x * DCP_THREADS) >> 5;
  DcpGuard guard;
  T km[DCP_NK];
  dcp_load_multipliers(km, dcp_km);
  for (long long w = warp; w < items; w += nwarps) {
    DcpItem it;
    it.in = p.ld[0];
    it.nz = p.nz;
    it.ny = p.ny;
    it.nx = p.nx;
    const long long yb = w / strips;
    it.x0 = (int)(w - yb * strips) * W;
    const int sg = (int)(yb / blocks);
    it.y0 = (int)(yb - (long long)sg * blocks) * (LY * CY);
    it.z0 = sg * p.seg;
    it.z1 = min(p.nz, it.z0 + p.seg);
    it.ring = (unsigned)__cvta_generic_to_shared(dcp_smem) + (threadIdx.x >> 5) * (R * PLANEB);
    const int col0 = it.x0 - HX + lane % LX * C, yl = it.y0 + lane / LX * CY;
    unsigned wm = 0u;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int x = col0 + c;
      wm |= x >= it.x0 && x < it.x0 + W && x < p.nx ? 1u << c : 0u;
    }
    auto output = [&](int z, const T (&v)[CY][C]) {
      long long gi = ((long long)z * p.ny + yl) * p.nx + col0;
#pragma unroll
      for (int r = 0; r < CY; ++r, gi += p.nx) {
        if (yl + r >= p.ny) break;
        T sv[DCP_ARR(DCP_NSTORE)][C];
#if DCP_POST
#pragma unroll
        for (int c = 0; c < C; ++c) {
          if (!((wm >> c) & 1u)) continue;
          T stv[DCP_ARR(DCP_NSTORE)], rv[DCP_ARR(DCP_NRED)];
          dcp_post(p, sc, gi + c, v[r][c], stv, rv);
#pragma unroll
          for (int s = 0; s < DCP_NSTORE; ++s) sv[s][c] = stv[s];
#pragma unroll
          for (int q = 0; q < DCP_NRED; ++q)
            acc[q] = dcp_red_comb(dcp_red_op(q), acc[q], dcp_red_lift(dcp_red_op(q), rv[q]));
        }
#else
#pragma unroll
        for (int c = 0; c < C; ++c) sv[0][c] = v[r][c];
#endif
#pragma unroll
        for (int s = 0; s < DCP_NSTORE; ++s) {
          typedef typename DcpAcc<V>::type A;
#pragma unroll
          for (int u = 0; u < C / V; ++u) {
            union { A a; T t[V]; } x;
#pragma unroll
            for (int e = 0; e < V; ++e) x.t[e] = sv[s][u * V + e];
            if ((wm >> (u * V)) & 1u) *reinterpret_cast<A*>(p.st[s] + gi + u * V) = x.a;
          }
        }
      }
    };
    // every column the strip reads lies inside the array (and the lanes'
    // outside a fixed ring)
    const int first = it.x0 - HX - C;
    if (first >= 0 && first + ROWE <= p.nx) dcp_column<false>(it, output, guard, km);
    else dcp_column<true>(it, output, guard, km);
  }
#if DCP_LAST && DCP_NRED > 0
  dcp_reduce_epilogue<T, DCP_NRED, DCP_THREADS>(acc, p.red_out, p.partials, p.ticket);
#endif
#if DCP_GUARD
  guard.flush(p.guard);
#endif
}
