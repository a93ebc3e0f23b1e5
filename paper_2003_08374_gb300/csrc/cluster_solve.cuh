// cluster_solve.cuh -- multigrid V-cycles and whole CG solves of small grids inside one
// thread-block cluster per domain (included by pressure.cu, inside namespace mdbs).
//
// A grid of a few thousand cells gives a kernel a few tenths of a microsecond of work, so
// run as launches its solve is launch and dependency latency: about 5 us for each of the
// eight kernels of a CG iteration and as many for a level's half sweeps.  Here the levels'
// iterates, right-hand sides and coefficients live in the distributed shared memory of a
// cluster for the kernel's whole life, and the phases of a V-cycle are separated by cluster
// barriers (levels spread over the CTAs), block barriers (levels in CTA 0 alone) or warp
// barriers (the smallest).
//
// What bounds a phase (measured on GB300, cycles): one FP64 instruction of a warp holds its
// quarter of the SM for 64, dependent or not and whatever the number of active lanes; a
// cluster barrier takes 400-500, a remote shared load 220, a local one 29, a block barrier
// 27, an FP64 division 1600, a square root 680.  So a level stays in one CTA until its FP64
// work costs more than the cluster barrier and the remote loads (kClSoloWork), colours are
// listed apart so that no lane idles, coefficients and neighbour addresses are read before
// the barrier of a phase, and scalars are formed by one warp.
//
// Every value is formed by the same operations in the same order as in the per-level
// launches (smooth_cell, resid_cell, the CG kernels and their reductions), so a solve here
// is bitwise the solve there.
//
// Layout.  CTA r of the cluster holds storage positions [r << shift, (r + 1) << shift) of a
// level; levels of little work sit in CTA 0.  The CG kernel's finest level is dealt out by
// the columns of the reductions instead (cl_owner), so that each CTA can run the chains of
// its columns.  Within the CTA the cells of colour 0 come
// first, then colour 1 (slots; ord maps a slot to its local position).  Each cell has its
// off-diagonal coefficients next to it (zero where there is no neighbour, whose product with
// the cell's own x then adds nothing) and the cluster addresses of its neighbours' x.

constexpr int kClThreads = 256;
constexpr int kClRow = kBlock;                 // cells of one reduction row
constexpr int kClSum = kClRow * kRepBig;       // cells of one partial sum: kRepBig rows
constexpr int kClMaxCtas = 16;                 // a non-portable cluster size
constexpr int kClCells = kClRow * kClMaxCtas;  // largest level a cluster takes
constexpr int kClRowsMax = 4;                  // rows' worth of cells a CTA of the CG kernel may hold
static_assert(kRepBig == 8 && kClRow == 256 && kClCells == 2 * kClSum, "cl_owner, total");
constexpr int kClSoloWork = 3072;              // cells x operations per update of a level kept in CTA 0
constexpr int kClSoloWork32 = 4096;            // (FP32: its shared memory, not its arithmetic, is what counts)
constexpr size_t kClSmemMax = 198 * 1024;      // dynamic shared memory (227 KB less the kernels' static part)
constexpr int kClWarp = 64;                    // levels up to this size run in one warp (32 cells of a colour)

// one level in the cluster's shared memory; the offsets are the same in every CTA
struct ClLevel {
  int cells, shift, solo;
  int lcol;      // log2 of the columns (of kClRow) a CTA holds of each row; -1: contiguous positions
  int here;      // cells in this CTA
  int red;       // of these, colour 0
  int most;      // the larger of its counts of the two colours
  int ne;        // neighbours per cell: 2, 4 or 6
  int cap;       // slots the arrays are sized for (stride of coef, nb and ch)
  int nch;       // residuals of the finer level that make up a right-hand side
  // shared addresses in this CTA (res: position order)
  unsigned x, b, res, dinv, diag, coef, nb, par, ch, ord;
};

__host__ __device__ __forceinline__ int ceil_log2(int v) {
  int s = 0;
  while ((1 << s) < v) s++;
  return s;
}
__host__ __device__ __forceinline__ unsigned cl_align(unsigned o) { return (o + 15u) & ~15u; }

// Shared-memory layout of a level of n cells in a cluster of ctas CTAs from offset o on;
// returns the end.  rows > 0: the CG kernel, rows * kClRow cells of the finest level (top) a
// CTA; where rows is more than one the SMs are shared out among many domains, and a level
// stays in CTA 0 only up to half the size.  finer_solo: the level above is in CTA 0, and so is this one.
// nch: children of a cell that the restriction sums (0 on the first level).
template <typename R>
__host__ __device__ inline unsigned cl_place(ClLevel& L, const int n[3], int nch, int ctas, int rows, bool top,
                                             bool finer_solo, unsigned o) {
  const int cells = n[0] * n[1] * n[2];
  L.nch = nch;
  L.cells = cells;
  L.ne = n[2] > 1 ? 6 : (n[1] > 1 ? 4 : 2);
  const bool fp64 = sizeof(R) == 8;
  const int row_cells = top ? rows * kClRow : 0, share = rows > 1 ? 2 : 1;
  if (row_cells > 0)
    L.solo = cells <= row_cells;
  else
    L.solo = ctas == 1 || finer_solo || share * cells * (L.ne + 1) <= (fp64 ? kClSoloWork : kClSoloWork32);
  L.lcol = row_cells > 0 && !L.solo ? ceil_log2(kClRow * rows / kRepBig) : -1;
  L.shift = L.solo ? ceil_log2(cells) : (row_cells > 0 ? ceil_log2(row_cells) : ceil_log2((cells + ctas - 1) / ctas));
  const int cap = (1 << L.shift) < cells ? (1 << L.shift) : cells;
  L.cap = cap;
  auto take = [&](unsigned bytes) {
    const unsigned at = o;
    o = cl_align(o + bytes);
    return at;
  };
  L.x = take(cap * sizeof(R));
  L.b = take(cap * sizeof(R));
  L.res = take(cap * sizeof(R));
  L.dinv = take(cap * sizeof(R));
  L.diag = take(cap * sizeof(R));
  L.coef = take(L.ne * cap * sizeof(R));
  L.nb = take(L.ne * cap * 4);
  L.par = take(cap * 4);        // cluster address of the parent cell's x
  L.ch = take(nch * cap * 4);   // cluster addresses of the children's residuals, in the restriction's order
  L.ord = take(cap * 2);
  return o;
}
// owner CTA and local index of storage position pos, and the position of (rank, local index).
// By columns: a partial sum covers kRepBig rows of kClRow positions, thread t of a block
// chains the products of its column t, and a warp then folds 32 columns; a CTA holds
// 32 rows of them (rows as in cl_place) of one partial sum.
__device__ __forceinline__ unsigned cl_owner(const ClLevel& L, unsigned pos) {
  return L.lcol < 0 ? pos >> L.shift : (pos / kClSum) * ((unsigned)kClRow >> L.lcol) + ((pos % kClRow) >> L.lcol);
}
__device__ __forceinline__ unsigned cl_local(const ClLevel& L, unsigned pos) {
  return L.lcol < 0 ? pos & ((1u << L.shift) - 1u)
                    : ((pos / kClRow % kRepBig) << L.lcol) + (pos & ((1u << L.lcol) - 1u));
}
__device__ __forceinline__ unsigned cl_position(const ClLevel& L, unsigned rank, unsigned e) {
  if (L.lcol < 0) return (rank << L.shift) + e;
  const unsigned per = (unsigned)kClRow >> L.lcol;
  return rank / per * kClSum + (e >> L.lcol) * kClRow + ((rank % per) << L.lcol) + (e & ((1u << L.lcol) - 1u));
}
// cells of CTA rank: its local indexes are 0 .. here - 1
__device__ __forceinline__ int cl_here(const ClLevel& L, unsigned rank) {
  const int cap = L.lcol < 0 ? 1 << L.shift : kRepBig << L.lcol;
  if (L.lcol < 0) {
    const int left = L.cells - (int)(rank << L.shift);
    return left <= 0 ? 0 : (left < cap ? left : cap);
  }
  const int per = kClRow >> L.lcol, cols = 1 << L.lcol;
  const int left = L.cells - (int)(rank / per) * kClSum;  // of this partial sum
  if (left <= 0) return 0;
  if (left >= kClSum) return cap;
  const int last = left % kClRow - (int)(rank % per) * cols;  // columns in the last, unfilled row
  return left / kClRow * cols + (last <= 0 ? 0 : (last < cols ? last : cols));
}
// children of a cell of a level coarsened along the axes cz; mask: colour 0 only
__host__ __device__ inline int cl_children(const int cz[3], int mask) {
  const int n = 1 << (cz[0] + cz[1] + cz[2]);
  return mask && n > 1 ? n / 2 : n;
}

// Shared memory by 32-bit address: this CTA's (sh_) or any CTA's of the cluster (cl_).  The
// loads clobber memory as the stores do: some of it (the level table, the exchanged sums) is
// also read or written by C++ statements, which the compiler may then not move past them.
__device__ __forceinline__ unsigned sh_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned cl_map(unsigned addr, unsigned rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void sh_ld(unsigned a, double& v) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory"); }
__device__ __forceinline__ void sh_ld(unsigned a, float& v) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory"); }
__device__ __forceinline__ unsigned sh_ldw(unsigned a) {
  unsigned v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ unsigned sh_ld16(unsigned a) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sh_st(unsigned a, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
__device__ __forceinline__ void sh_st(unsigned a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void sh_st(unsigned a, unsigned v) { asm volatile("st.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory"); }
__device__ __forceinline__ void sh_st16(unsigned a, unsigned v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}
// predicated stores: no branch around them, which costs as much as a phase's loads
__device__ __forceinline__ void sh_st_if(unsigned a, double v, bool ok) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p st.shared.f64 [%0], %1;\n}\n" ::"r"(a), "d"(v), "r"((unsigned)ok) : "memory");
}
__device__ __forceinline__ void sh_st_if(unsigned a, float v, bool ok) {
  asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %2, 0;\n @p st.shared.f32 [%0], %1;\n}\n" ::"r"(a), "f"(v), "r"((unsigned)ok) : "memory");
}
__device__ __forceinline__ void cl_ld(unsigned a, double& v) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ void cl_ld(unsigned a, float& v) {
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
}
__device__ __forceinline__ unsigned cl_ld16(unsigned a) {
  unsigned short v;
  asm volatile("ld.shared::cluster.u16 %0, [%1];" : "=h"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void cl_st(unsigned a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// Who runs a phase: the whole cluster, CTA 0, or its first warp.  A phase reads what is
// static, waits for the phases before it (begin), works, and signals its end: between
// phases of the cluster that is an arrival at the cluster barrier, which the next phase
// (or whoever reads the result) waits for.
//
// Who runs a phase is a template parameter, and every phase is inlined.  As functions of
// their own they were no faster, and gave wrong results, not the same ones each time, with
// four rows a CTA in FP64 on 9 x 20 x 11 cells.  The cause of that is not known: reading the
// phases' barriers for that shape showed none, and the loads above did not clobber memory
// then.  The inlined form is compared bit for bit with the launches over shapes of every row
// count.  The phases take shared addresses (lv: a ClLevel) and copy no table to local memory;
// what the four-row FP64 kernel holds there is 136 bytes of spilled registers.
enum { kByCluster = 0, kByBlock = 1, kByWarp = 2 };
template <int KIND>
__device__ __forceinline__ void cl_begin() {
  if constexpr (KIND == kByCluster)
    cl_wait();
  else if constexpr (KIND == kByBlock)
    __syncthreads();
  else
    __syncwarp();
}
template <int KIND>
__device__ __forceinline__ void cl_end() {
  if constexpr (KIND == kByCluster) cl_arrive();
}
template <int KIND>
constexpr unsigned kClStep = KIND == kByWarp ? 32u : (unsigned)kClThreads;
// field of the ClLevel at shared address lv
#define CL_F(lv, field) sh_ldw((lv) + (unsigned)offsetof(ClLevel, field))

template <typename R>
struct Cl {
  unsigned lv;      // shared address of the level table, index = multigrid level
  unsigned rank;    // CTA rank in the cluster
  unsigned cinv;    // shared address of the coarsest inverse
  __device__ __forceinline__ unsigned level(int l) const { return lv + (unsigned)l * (unsigned)sizeof(ClLevel); }
};

// One red-black half sweep over this CTA's cells of colour col (zero: the other colour's x
// is taken as 0).
template <typename R, int KIND, int NE>
__device__ __forceinline__ void cl_half_ne(unsigned lv, int col, int zero) {
  constexpr unsigned W = sizeof(R);
  const unsigned cap = CL_F(lv, cap), red = CL_F(lv, red), here = CL_F(lv, here);
  const unsigned x = CL_F(lv, x), b = CL_F(lv, b), dinv = CL_F(lv, dinv), cf = CL_F(lv, coef), nb = CL_F(lv, nb);
  const unsigned last = col ? here : red, step = kClStep<KIND>;
  unsigned e = (col ? red : 0u) + threadIdx.x;
  unsigned a[NE] = {};
  R k[NE] = {}, di = R(0);
  auto fetch = [&] {
    sh_ld(dinv + e * W, di);
    if (!zero) {
#pragma unroll
      for (int d = 0; d < NE; d++) {
        a[d] = sh_ldw(nb + (d * cap + e) * 4u);
        sh_ld(cf + (d * cap + e) * W, k[d]);
      }
    }
  };
  if (e < last) fetch();
  cl_begin<KIND>();
  while (e < last) {
    R v, xn[NE];
    sh_ld(b + e * W, v);
    if (!zero) {
#pragma unroll
      for (int d = 0; d < NE; d++) cl_ld(a[d], xn[d]);
#pragma unroll
      for (int d = 0; d < NE; d++) v = fma_r(k[d], xn[d], v);
    }
    sh_st(x + e * W, v * di);
    e += step;
    if (e < last) fetch();
  }
  cl_end<KIND>();
}
template <typename R, int KIND>
__device__ __forceinline__ void cl_half(unsigned lv, int col, int zero) {
  const unsigned ne = CL_F(lv, ne);
  if (ne == 6)
    cl_half_ne<R, KIND, 6>(lv, col, zero);
  else if (ne == 4)
    cl_half_ne<R, KIND, 4>(lv, col, zero);
  else
    cl_half_ne<R, KIND, 2>(lv, col, zero);
}

// residual b - A x of this CTA's cells (mask: colour 0 only), into res
template <typename R, int KIND, int NE>
__device__ __forceinline__ void cl_resid_ne(unsigned lv, int mask) {
  constexpr unsigned W = sizeof(R);
  const unsigned cap = CL_F(lv, cap), last = mask ? CL_F(lv, red) : CL_F(lv, here), step = kClStep<KIND>;
  const unsigned x = CL_F(lv, x), b = CL_F(lv, b), dg = CL_F(lv, diag), cf = CL_F(lv, coef), nb = CL_F(lv, nb);
  const unsigned res = CL_F(lv, res), ord = CL_F(lv, ord);
  unsigned e = threadIdx.x, pos = 0;
  unsigned a[NE] = {};
  R k[NE] = {}, dv = R(0), bv = R(0);
  auto fetch = [&] {
    pos = sh_ld16(ord + e * 2u);
    sh_ld(dg + e * W, dv);
#pragma unroll
    for (int d = 0; d < NE; d++) {
      a[d] = sh_ldw(nb + (d * cap + e) * 4u);
      sh_ld(cf + (d * cap + e) * W, k[d]);
    }
  };
  if (e < last) fetch();
  cl_begin<KIND>();
  while (e < last) {
    R xn[NE], xo;
    sh_ld(b + e * W, bv);
    sh_ld(x + e * W, xo);
#pragma unroll
    for (int d = 0; d < NE; d++) cl_ld(a[d], xn[d]);
    R v = R(0);
#pragma unroll
    for (int d = 0; d < NE; d++) v = fma_r(k[d], xn[d], v);
    sh_st(res + pos * W, bv - (mul_r(dv, xo) - v));
    e += step;
    if (e < last) fetch();
  }
  cl_end<KIND>();
}
template <typename R, int KIND>
__device__ __forceinline__ void cl_resid(unsigned lv, int mask) {
  const unsigned ne = CL_F(lv, ne);
  if (ne == 6)
    cl_resid_ne<R, KIND, 6>(lv, mask);
  else if (ne == 4)
    cl_resid_ne<R, KIND, 4>(lv, mask);
  else
    cl_resid_ne<R, KIND, 2>(lv, mask);
}

// right-hand side of the level at lv: its children's residuals summed in the order of
// b_resid_restrict; fold: also its zero-guess colour-0 update.  Lanes beyond the cells
// repeat cell 0 and store nothing; warps beyond them do nothing.
template <typename R, int KIND, int NCH>
__device__ __forceinline__ void cl_gather_n(unsigned lv, int fold) {
  constexpr unsigned W = sizeof(R);
  const unsigned cap = CL_F(lv, cap), here = CL_F(lv, here), red = CL_F(lv, red);
  const unsigned b = CL_F(lv, b), x = CL_F(lv, x), dinv = CL_F(lv, dinv), ch = CL_F(lv, ch), step = kClStep<KIND>;
  const unsigned lane = threadIdx.x & 31u;
  unsigned a[NCH], e = 0;
  R di = R(0);
  bool ok = false;
  auto fetch = [&](unsigned base) {
    ok = base + lane < here;
    e = ok ? base + lane : 0u;
#pragma unroll
    for (int q = 0; q < NCH; q++) a[q] = sh_ldw(ch + ((unsigned)q * cap + e) * 4u);
    sh_ld(dinv + e * W, di);
  };
  unsigned base = threadIdx.x - lane;
  if (base < here) fetch(base);
  cl_begin<KIND>();
  while (base < here) {
    R r[NCH];
#pragma unroll
    for (int q = 0; q < NCH; q++) cl_ld(a[q], r[q]);
    R s = R(0);
#pragma unroll
    for (int q = 0; q < NCH; q++) s += r[q];
    sh_st_if(b + e * W, s, ok);
    if (fold && base < red) sh_st_if(x + e * W, s * di, ok && e < red);
    base += step;
    if (base < here) fetch(base);
  }
  cl_end<KIND>();
}
template <typename R, int KIND>
__device__ __forceinline__ void cl_gather(unsigned lv, int fold) {
  const unsigned n = CL_F(lv, nch);
  if (n == 1)
    cl_gather_n<R, KIND, 1>(lv, fold);
  else if (n == 2)
    cl_gather_n<R, KIND, 2>(lv, fold);
  else if (n == 4)
    cl_gather_n<R, KIND, 4>(lv, fold);
  else
    cl_gather_n<R, KIND, 8>(lv, fold);
}

// x += the parents' x; only colour 0 when a half sweep of colour 1 follows (that sweep
// reads colour 0 alone and overwrites colour 1)
template <typename R, int KIND>
__device__ __forceinline__ void cl_prolong(unsigned lv, int red_only) {
  constexpr unsigned W = sizeof(R);
  const unsigned last = red_only ? CL_F(lv, red) : CL_F(lv, here), x = CL_F(lv, x), par = CL_F(lv, par);
  const unsigned step = kClStep<KIND>;
  unsigned e = threadIdx.x;
  cl_begin<KIND>();
  for (; e < last; e += step) {
    R xv, ev;
    const unsigned a = sh_ldw(par + e * 4u);
    sh_ld(x + e * W, xv);
    cl_ld(a, ev);
    sh_st(x + e * W, xv + ev);
  }
  cl_end<KIND>();
}

template <typename R, int KIND>
__device__ __forceinline__ void cl_zero(unsigned lv) {
  cl_begin<KIND>();
  const unsigned here = CL_F(lv, here), x = CL_F(lv, x), step = kClStep<KIND>;
  for (unsigned e = threadIdx.x; e < here; e += step) sh_st(x + e * (unsigned)sizeof(R), R(0));
  cl_end<KIND>();
}

// exact coarsest solve, one row of the inverse a thread (b and x in storage order)
template <typename R>
__device__ __forceinline__ void coarse_solve(const R* cinv, const R* b, R* x, int n, unsigned t, unsigned nt) {
  for (int i = (int)t; i < n; i += (int)nt) {
    R v = R(0);
    for (int j = 0; j < n; j++) v = fma_r(cinv[i * n + j], b[j], v);
    x[i] = v;
  }
}

// the same on the slots of the coarsest level; row i of the inverse starts at i (n + 1), so
// that the rows of a warp fall into different banks
template <typename R, int KIND>
__device__ __forceinline__ void cl_coarse(unsigned lv, unsigned cinv) {
  constexpr unsigned W = sizeof(R);
  const unsigned n = CL_F(lv, cells), b = CL_F(lv, b), x = CL_F(lv, x), res = CL_F(lv, res), ord = CL_F(lv, ord);
  const unsigned step = kClStep<KIND>;
  cl_begin<KIND>();
  // b to position order (res is free on the coarsest level)
  for (unsigned e = threadIdx.x; e < n; e += step) {
    R v;
    sh_ld(b + e * W, v);
    sh_st(res + sh_ld16(ord + e * 2u) * W, v);
  }
  cl_begin<KIND>();
  for (unsigned e = threadIdx.x; e < n; e += step) {
    const unsigned row = cinv + sh_ld16(ord + e * 2u) * (n + 1) * W;
    R v = R(0);
    unsigned j = 0;
    for (; j + 8 <= n; j += 8) {  // eight products' loads in flight: the chain is the fma's 64 cycles each
      R m[8], bj[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        sh_ld(row + (j + q) * W, m[q]);
        sh_ld(res + (j + q) * W, bj[q]);
      }
#pragma unroll
      for (int q = 0; q < 8; q++) v = fma_r(m[q], bj[q], v);
    }
    for (; j < n; j++) {
      R m, bj;
      sh_ld(row + j * W, m);
      sh_ld(res + j * W, bj);
      v = fma_r(m, bj, v);
    }
    sh_st(x + e * W, v);
  }
  cl_end<KIND>();
}

// most cells of one colour a thread may have in a descent or ascent: two with two neighbours
// each (the first coarse levels of a column), else one
__host__ __device__ constexpr int cl_per_thread(int ne) { return ne == 2 ? 2 : 1; }

// A level's whole descent or ascent where every thread has at most cl_per_thread cells of a colour
// (all levels but a few): coefficients, addresses and right-hand sides stay in registers
// from one phase to the next, and a phase is a barrier, one round of loads, the fma chain
// and a store.  The separate phases fetch them again each time: 640-830 cycles a half sweep
// of one warp, of which 200-450 are FP64.
// Lanes without a cell repeat slot 0 and store nothing; warps without one do nothing.
template <typename R, int NE>
struct ClCell {
  unsigned e, nb[NE];
  R k[NE], di;
  bool ok, warp;  // this thread, this warp has a cell
  __device__ __forceinline__ void fetch(unsigned from, unsigned last, unsigned cap, unsigned dinv, unsigned cf, unsigned na) {
    constexpr unsigned W = sizeof(R);
    const unsigned slot = from + threadIdx.x;
    ok = slot < last;
    warp = from + (threadIdx.x & ~31u) < last;
    e = ok ? slot : 0u;
    sh_ld(dinv + e * W, di);
#pragma unroll
    for (int d = 0; d < NE; d++) {
      nb[d] = sh_ldw(na + (d * cap + e) * 4u);
      sh_ld(cf + (d * cap + e) * W, k[d]);
    }
  }
  __device__ __forceinline__ R sum(R v) const {
    R xn[NE];
#pragma unroll
    for (int d = 0; d < NE; d++) cl_ld(nb[d], xn[d]);
#pragma unroll
    for (int d = 0; d < NE; d++) v = fma_r(k[d], xn[d], v);
    return v;
  }
};

template <typename R, int KIND, int NE>
__device__ __forceinline__ void cl_down_one(unsigned lv, int nu1, int folded) {
  constexpr unsigned W = sizeof(R);
  constexpr int M = cl_per_thread(NE);
  const unsigned cap = CL_F(lv, cap), red = CL_F(lv, red), here = CL_F(lv, here);
  const unsigned x = CL_F(lv, x), b = CL_F(lv, b), dinv = CL_F(lv, dinv), cf = CL_F(lv, coef), nb = CL_F(lv, nb);
  const unsigned diag = CL_F(lv, diag), rs = CL_F(lv, res), ord = CL_F(lv, ord);
  ClCell<R, NE> c0[M], c1[M];
  R dg[M], b0[M], b1[M];
  unsigned res[M];
#pragma unroll
  for (int m = 0; m < M; m++) {
    c0[m].fetch(m * kClStep<KIND>, red, cap, dinv, cf, nb);
    c1[m].fetch(red + m * kClStep<KIND>, here, cap, dinv, cf, nb);
    sh_ld(diag + c0[m].e * W, dg[m]);
    res[m] = rs + sh_ld16(ord + c0[m].e * 2u) * W;
  }
  cl_begin<KIND>();
#pragma unroll
  for (int m = 0; m < M; m++) {
    sh_ld(b + c0[m].e * W, b0[m]);
    sh_ld(b + c1[m].e * W, b1[m]);
  }
  if (!folded) {
#pragma unroll
    for (int m = 0; m < M; m++)
      if (c0[m].warp) sh_st_if(x + c0[m].e * W, b0[m] * c0[m].di, c0[m].ok);
    cl_end<KIND>();
    cl_begin<KIND>();
  }
  for (int it = 0;; it++) {
#pragma unroll
    for (int m = 0; m < M; m++)
      if (c1[m].warp) sh_st_if(x + c1[m].e * W, c1[m].sum(b1[m]) * c1[m].di, c1[m].ok);
    cl_end<KIND>();
    cl_begin<KIND>();
    if (it + 1 >= nu1) break;
#pragma unroll
    for (int m = 0; m < M; m++)
      if (c0[m].warp) sh_st_if(x + c0[m].e * W, c0[m].sum(b0[m]) * c0[m].di, c0[m].ok);
    cl_end<KIND>();
    cl_begin<KIND>();
  }
#pragma unroll
  for (int m = 0; m < M; m++)
    if (c0[m].warp) {
      R xo;
      sh_ld(x + c0[m].e * W, xo);
      const R v = c0[m].sum(R(0));
      sh_st_if(res[m], b0[m] - (mul_r(dg[m], xo) - v), c0[m].ok);
    }
  cl_end<KIND>();
}

template <typename R, int KIND, int NE>
__device__ __forceinline__ void cl_up_one(unsigned lv, int nu2) {
  constexpr unsigned W = sizeof(R);
  constexpr int M = cl_per_thread(NE);
  const unsigned cap = CL_F(lv, cap), red = CL_F(lv, red), here = CL_F(lv, here);
  const unsigned x = CL_F(lv, x), b = CL_F(lv, b), dinv = CL_F(lv, dinv), cf = CL_F(lv, coef), nb = CL_F(lv, nb);
  const unsigned pa = CL_F(lv, par);
  ClCell<R, NE> c0[M], c1[M];
  R b0[M], b1[M], xo[M];
  unsigned par[M];
#pragma unroll
  for (int m = 0; m < M; m++) {
    c0[m].fetch(m * kClStep<KIND>, red, cap, dinv, cf, nb);
    c1[m].fetch(red + m * kClStep<KIND>, here, cap, dinv, cf, nb);
    sh_ld(b + c0[m].e * W, b0[m]);
    par[m] = sh_ldw(pa + c0[m].e * 4u);
    sh_ld(b + c1[m].e * W, b1[m]);
  }
  cl_begin<KIND>();
#pragma unroll
  for (int m = 0; m < M; m++)
    if (c0[m].warp) {
      R ev;
      cl_ld(par[m], ev);
      sh_ld(x + c0[m].e * W, xo[m]);
      sh_st_if(x + c0[m].e * W, xo[m] + ev, c0[m].ok);
    }
  cl_end<KIND>();
  for (int it = 0; it < nu2; it++) {
    cl_begin<KIND>();
#pragma unroll
    for (int m = 0; m < M; m++)
      if (c1[m].warp) sh_st_if(x + c1[m].e * W, c1[m].sum(b1[m]) * c1[m].di, c1[m].ok);
    cl_end<KIND>();
    cl_begin<KIND>();
#pragma unroll
    for (int m = 0; m < M; m++)
      if (c0[m].warp) sh_st_if(x + c0[m].e * W, c0[m].sum(b0[m]) * c0[m].di, c0[m].ok);
    cl_end<KIND>();
  }
}

template <int KIND>
__device__ __forceinline__ bool cl_fits(unsigned lv) {
  return CL_F(lv, most) <= kClStep<KIND> * (unsigned)cl_per_thread((int)CL_F(lv, ne));
}

// pre-smoothing and residual of a level (its b is complete; folded: its zero-guess
// colour-0 update came with b)
template <typename R, int KIND>
__device__ __forceinline__ void cl_down(unsigned lv, int nu1, int folded) {
  if (nu1 > 0 && cl_fits<KIND>(lv)) {
    const unsigned ne = CL_F(lv, ne);
    if (ne == 6)
      cl_down_one<R, KIND, 6>(lv, nu1, folded);
    else if (ne == 4)
      cl_down_one<R, KIND, 4>(lv, nu1, folded);
    else
      cl_down_one<R, KIND, 2>(lv, nu1, folded);
    return;
  }
  if (nu1 == 0) cl_zero<R, KIND>(lv);
  for (int h = folded ? 1 : 0; h < 2 * nu1; h++) cl_half<R, KIND>(lv, h & 1, h == 0);
  cl_resid<R, KIND>(lv, nu1 > 0 ? 1 : 0);
}
template <typename R, int KIND>
__device__ __forceinline__ void cl_up(unsigned lv, int nu2) {
  if (nu2 > 0 && cl_fits<KIND>(lv)) {
    const unsigned ne = CL_F(lv, ne);
    if (ne == 6)
      cl_up_one<R, KIND, 6>(lv, nu2);
    else if (ne == 4)
      cl_up_one<R, KIND, 4>(lv, nu2);
    else
      cl_up_one<R, KIND, 2>(lv, nu2);
    return;
  }
  cl_prolong<R, KIND>(lv, nu2 > 0 ? 1 : 0);
  for (int h = 0; h < 2 * nu2; h++) cl_half<R, KIND>(lv, 1 - (h & 1), 0);
}

// the levels in CTA 0 from level l0 on, called by all its threads; ends with a block barrier
template <typename R>
__device__ __forceinline__ void cl_solo(const Cl<R>& c, int l0, int nlev, int nu1, int nu2, int cs, int folded) {
  const int mask = nu1 > 0 ? 1 : 0, lc = nlev - 1;
  int lw = l0;  // first level of the single warp
  while (lw < lc && CL_F(c.level(lw), cells) > kClWarp) lw++;
  for (int l = l0; l < lw; l++) {
    cl_down<R, kByBlock>(c.level(l), nu1, l == l0 ? folded : mask);
    cl_gather<R, kByBlock>(c.level(l + 1), mask);
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    for (int l = lw; l < lc; l++) {
      cl_down<R, kByWarp>(c.level(l), nu1, l == l0 ? folded : mask);
      cl_gather<R, kByWarp>(c.level(l + 1), mask);
    }
    for (int h = 0; h < 2 * cs; h++) cl_half<R, kByWarp>(c.level(lc), h & 1, h == 0);
    for (int h = 0; h < 2 * cs; h++) cl_half<R, kByWarp>(c.level(lc), 1 - (h & 1), 0);
  }
  if (cs == 0) {
    const bool wide = CL_F(c.level(lc), cells) > 32;
    if (wide)
      cl_coarse<R, kByBlock>(c.level(lc), c.cinv);
    else if (threadIdx.x < 32)
      cl_coarse<R, kByWarp>(c.level(lc), c.cinv);
    if (wide) __syncthreads();
  }
  if (threadIdx.x < 32)
    for (int l = lc - 1; l >= lw; l--) cl_up<R, kByWarp>(c.level(l), nu2);
  for (int l = lw - 1; l >= l0; l--) cl_up<R, kByBlock>(c.level(l), nu2);
  __syncthreads();
}

// The V-cycle from level first down, called by every thread of the cluster; b of level
// first is in its owners' slots.  When level first is spread over the CTAs the caller has
// arrived at the cluster barrier, and waits for the last half sweep's arrival; otherwise
// everything happens in CTA 0 between block barriers.
template <typename R>
__device__ __forceinline__ void cl_vcycle(Cl<R> c, int first, int nlev, int nu1, int nu2, int cs) {
  const int mask = nu1 > 0 ? 1 : 0;
  int ls = first;  // first level in CTA 0
  while (!CL_F(c.level(ls), solo)) ls++;
  for (int l = first; l < ls; l++) {
    cl_down<R, kByCluster>(c.level(l), nu1, l == first ? 0 : mask);
    if (l + 1 < ls) cl_gather<R, kByCluster>(c.level(l + 1), mask);
  }
  if (ls > first) cl_wait();
  if (c.rank == 0) {
    if (ls > first) cl_gather<R, kByBlock>(c.level(ls), mask);
    cl_solo<R>(c, ls, nlev, nu1, nu2, cs, ls > first ? mask : 0);
  }
  if (ls > first) cl_arrive();
  for (int l = ls - 1; l >= first; l--) cl_up<R, kByCluster>(c.level(l), nu2);
}

// Level table, coefficients, slots and neighbour addresses of levels first .. nlev - 1.
// Reads only what the operator build wrote (static during a solve).  Contains a cluster
// barrier; ends with a block barrier.
// sm: this CTA's dynamic shared memory; *end: its first free byte afterwards; mask: the
// restriction sums colour 0 only.
template <typename R>
__device__ void cl_setup(Cl<R>& c, ClLevel* lv, Level<R>* gl, unsigned sm, const CgDom& G, int first, int nlev,
                         int ctas, int rows, int mask, unsigned* end) {
  constexpr unsigned W = sizeof(R);
  __shared__ unsigned s_end, s_zero;
  __shared__ int s_off[kMaxLevels + 1];            // this CTA's cells of the levels before
  __shared__ int s_count[2][kMaxLevels];           // slots of each colour given out
  const unsigned tid = threadIdx.x;
  // the level views to shared memory: a cluster barrier's acquire empties L1
  for (int l = first + (int)tid; l < nlev; l += kClThreads) gl[l] = levels_of<R>(G)[l];
  __syncthreads();
  if (tid == 0) {
    unsigned o = sm;
    int at = 0;
    for (int l = first; l < nlev; l++) {
      o = cl_place<R>(lv[l], gl[l].n, l > first ? cl_children(gl[l].cz, mask) : 0, ctas, rows, l == first,
                      l > first && lv[l - 1].solo, o);
      ClLevel& L = lv[l];
      L.here = cl_here(L, c.rank);
      s_off[l] = at;
      at += L.here;
      s_count[0][l] = s_count[1][l] = 0;
    }
    s_off[nlev] = at;
    s_zero = o;
    s_end = o + 16;
    sh_st(o, 0.0);  // what a cell with fewer children adds
  }
  __syncthreads();
  const int total = s_off[nlev];
  // slots, in any order within a colour (no value depends on it): colour 0 from the bottom,
  // colour 1 from the top; the slot of each position goes to res until the barrier
  for (int f = (int)tid; f < total; f += kClThreads) {
    int l = first;
    while (f >= s_off[l + 1]) l++;
    const ClLevel& L = lv[l];
    const unsigned e = (unsigned)(f - s_off[l]);
    int q[3];
    decode_pos(gl[l], (long long)cl_position(L, c.rank, e), q[0], q[1], q[2]);
    const int col = (q[0] + q[1] + q[2]) & 1;
    const int k = atomicAdd(&s_count[col][l], 1);
    const unsigned slot = (unsigned)(col ? L.here - 1 - k : k);
    sh_st16(L.ord + slot * 2u, e);
    sh_st16(L.res + e * W, slot);
    sh_st(L.x + slot * W, R(0));  // a missing neighbour's product is 0 times this
  }
  cl_arrive();
  cl_wait();
  if ((int)tid >= first && (int)tid < nlev) {
    const int r = s_count[0][tid], k = lv[tid].here - r;
    lv[tid].red = r;
    lv[tid].most = r > k ? r : k;
  }
  for (int f = (int)tid; f < total; f += kClThreads) {
    int l = first;
    while (f >= s_off[l + 1]) l++;
    const ClLevel& L = lv[l];
    const Level<R>& A = gl[l];
    const unsigned e = (unsigned)(f - s_off[l]), pos = cl_position(L, c.rank, e);
    const unsigned cap = (unsigned)L.cap, slot = sh_ld16(L.res + e * W);
    int q[3];
    decode_pos(A, (long long)pos, q[0], q[1], q[2]);
    R k[6];
    unsigned a[6];
    const R di = A.dinv[pos], dg = A.diag[pos];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const bool has_lo = q[d] > 0, has_hi = q[d] + 1 < A.n[d];
      a[2 * d] = has_lo ? lo_pos(A.n, q, pos, d) : pos;
      a[2 * d + 1] = has_hi ? hi_pos(A.n, q, pos, d) : pos;
      k[2 * d] = has_lo ? tcoef(A, d, a[2 * d]) : R(0);
      k[2 * d + 1] = has_hi ? tcoef(A, d, pos) : R(0);
    }
    sh_st(L.dinv + slot * W, di);
    sh_st(L.diag + slot * W, dg);
#pragma unroll
    for (int d = 0; d < 6; d++)
      if (d < L.ne) {
        const unsigned r = cl_owner(L, a[d]), s = cl_ld16(cl_map(L.res + cl_local(L, a[d]) * W, r));
        sh_st(L.nb + (d * cap + slot) * 4u, cl_map(L.x + s * W, r));
        sh_st(L.coef + (d * cap + slot) * W, k[d]);
      }
    if (l + 1 < nlev) {
      const Level<R>& Co = gl[l + 1];
      const ClLevel& N = lv[l + 1];
      const unsigned pp =
          lpos(Co.n, Co.cz[0] ? q[0] >> 1 : q[0], Co.cz[1] ? q[1] >> 1 : q[1], Co.cz[2] ? q[2] >> 1 : q[2]);
      const unsigned r = cl_owner(N, pp), s = cl_ld16(cl_map(N.res + cl_local(N, pp) * W, r));
      sh_st(L.par + slot * 4u, cl_map(N.x + s * W, r));
    }
    if (l > first) {
      const Level<R>& Fi = gl[l - 1];
      const ClLevel& F = lv[l - 1];
      int lo[3], hi[3], k = 0;
      for (int d = 0; d < 3; d++) {
        lo[d] = A.cz[d] ? 2 * q[d] : q[d];
        hi[d] = A.cz[d] && 2 * q[d] + 1 < Fi.n[d] ? 2 * q[d] + 1 : lo[d];
      }
      for (int z = lo[2]; z <= hi[2]; z++)
        for (int y = lo[1]; y <= hi[1]; y++)
          for (int x = lo[0]; x <= hi[0]; x++) {
            if (mask && ((x + y + z) & 1)) continue;
            const unsigned p = lpos(Fi.n, x, y, z);
            sh_st(L.ch + (k * cap + slot) * 4u, cl_map(F.res + cl_local(F, p) * W, cl_owner(F, p)));
            k++;
          }
      for (; k < L.nch; k++) sh_st(L.ch + (k * cap + slot) * 4u, cl_map(s_zero, c.rank));
    }
  }
  const int n = (int)gl[nlev - 1].cells;
  const unsigned cv = s_end;
  c.cinv = cv;
  if (c.rank == 0) {
    const R* g = coarse_inverse_of<R>(G);
    for (int e = (int)tid; e < n * n; e += kClThreads) sh_st(cv + (unsigned)(e / n * (n + 1) + e % n) * W, g[e]);
  }
  *end = cl_align(cv + (unsigned)(n * (n + 1)) * W);
  __syncthreads();
}

// dynamic shared memory of levels first .. nlev - 1 (and of the CG kernel's vector)
template <typename R>
inline size_t cl_bytes(const Level<R>* gl, int first, int nlev, int ctas, int rows, int mask) {
  unsigned o = 0;
  ClLevel L{};
  for (int l = first; l < nlev; l++)
    o = cl_place<R>(L, gl[l].n, l > first ? cl_children(gl[l].cz, mask) : 0, ctas, rows, l == first,
                    l > first && L.solo, o);
  o += 16;
  const unsigned n = (unsigned)gl[nlev - 1].cells;
  return cl_align(o + n * (n + 1) * (unsigned)sizeof(R)) + (unsigned)(rows * kClRow) * 8u;
}

// ---- the tail levels of a V-cycle, one cluster per domain (idx: the domains)
template <typename R>
__global__ void __launch_bounds__(kClThreads, 2)
    k_tail_cluster(const CgDom* __restrict__ CG, const int* __restrict__ idx, int ctas, int nu1, int nu2, int cs) {
  extern __shared__ __align__(16) unsigned char cl_sm[];
  __shared__ ClLevel lv[kMaxLevels];
  __shared__ Level<R> gl[kMaxLevels];
  const CgDom& G = CG[idx[blockIdx.x / ctas]];
  Cl<R> c{sh_addr(lv), blockIdx.x % ctas, 0u};
  unsigned end;
  const int first = G.first, nlev = G.nlev;
  // Before the wait on the preceding kernel (a restriction or a half sweep, which may not have
  // waited itself): everything the setup reads was written by the operator's build, which had
  // completed before any kernel of the loop started (MDBS_PDL_TRIGGER).
  cl_setup<R>(c, lv, gl, sh_addr(cl_sm), G, first, nlev, ctas, 0, nu1 > 0 ? 1 : 0, &end);
  MDBS_DEPENDENT_ENTRY();
  // every thread of the cluster has left the setup's remote reads of res behind
  cl_arrive();
  cl_wait();
  if (G.scal[kCond] == 0.0) return;  // the same for the whole cluster
  const ClLevel& L = lv[first];
  const unsigned p0 = c.rank << L.shift;
  for (int e = (int)threadIdx.x; e < L.here; e += kClThreads)
    sh_st(L.b + e * (unsigned)sizeof(R), gl[first].b[p0 + sh_ld16(L.ord + e * 2u)]);
  __syncthreads();
  if (!L.solo) cl_arrive();
  cl_vcycle(c, first, nlev, nu1, nu2, cs);
  if (!L.solo) cl_wait();  // the last half sweep; no CTA leaves while another may read its shared memory
  for (int e = (int)threadIdx.x; e < L.here; e += kClThreads) {
    R v;
    sh_ld(L.x + e * (unsigned)sizeof(R), v);
    gl[first].x[p0 + sh_ld16(L.ord + e * 2u)] = v;
  }
}

// ---- a whole CG solve, one cluster per domain: the loop of pressure_solve for a domain
// whose finest level has at most kClCells cells and lies in the tail.  A CTA holds
// ROWS * kClRow cells, ROWS of them a thread: whole columns of the batched kernels'
// reductions, whose chains and trees it runs in their order.
template <typename R, int ROWS>
__global__ void __launch_bounds__(kClThreads, 1)
    k_cg_cluster(const StepDom* __restrict__ D, const CgDom* __restrict__ CG, const int* __restrict__ idx, int ctas,
                 int nu1, int nu2, int cs, double tol, int max_it, int early) {
  constexpr bool kFlex = std::is_same<R, float>::value;
  constexpr unsigned W = sizeof(R);
  extern __shared__ __align__(16) unsigned char cl_sm[];
  __shared__ ClLevel lv[kMaxLevels];
  __shared__ Level<R> gl[kMaxLevels];
  constexpr int kFactors = kFlex ? 3 : 2, kCols = 32 * ROWS;
  __shared__ double s_fac[kFactors][ROWS * kClThreads];
  __shared__ double s_part[2][2][kClMaxCtas];  // [exchange parity][sum][32 columns of a partial sum]
  __shared__ double s_scal[4];                 // beta, alpha, done
  const CgDom& G = CG[idx[blockIdx.x / ctas]];
  const StepDom& S = D[idx[blockIdx.x / ctas]];
  Cl<R> c{sh_addr(lv), blockIdx.x % ctas, 0u};
  unsigned end;
  const int nlev = G.nlev;
  // A step's first solve waits here: the operator's build may be among the kernels it follows
  // (the branch it runs on joins ahead of this kernel, and a captured join can be a
  // programmatic dependency like any other).  In the later ones, which follow the first, the
  // setup overlaps the preceding kernel (another size's solve among them); all it reads is the
  // operator.
  if (!early) MDBS_PDL_WAIT();
  cl_setup<R>(c, lv, gl, sh_addr(cl_sm), G, 0, nlev, ctas, ROWS, nu1 > 0 ? 1 : 0, &end);
  const unsigned db = end;  // the vector A is applied to, exchanged through the cluster

  const int n = (int)S.P.cells;
  const ClLevel& L0 = lv[0];
  const bool solo0 = L0.solo;
  const unsigned t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int slots = solo0 ? 1 : (n + kClSum - 1) / kClSum * (kClRow / 32);  // of s_part
  const int ne = S.P.n[2] > 1 ? 6 : (S.P.n[1] > 1 ? 4 : 2);
  // this thread's cells: operator rows, vectors, slots and the addresses of their neighbours
  bool in[ROWS];
  double T[ROWS][6], dg[ROWS], bc[ROWS], p[ROWS], r[ROWS], dval[ROWS], qval[ROWS];
  unsigned na[ROWS][6], nat[ROWS], slot[ROWS];
#pragma unroll
  for (int w = 0; w < ROWS; w++) {
    const unsigned e = w * kClThreads + t, pos = cl_position(L0, c.rank, e);
    in[w] = (int)e < L0.here;
    dg[w] = bc[w] = p[w] = dval[w] = qval[w] = 0.0;
    nat[w] = slot[w] = 0;
    for (int d = 0; d < 6; d++) {
      T[w][d] = 0.0;
      na[w][d] = db;
    }
    if (!in[w]) continue;
    int q[3];
    decode_pos(S.P, (long long)pos, q[0], q[1], q[2]);
    nat[w] = (unsigned)q[0] + (unsigned)S.P.n[0] * ((unsigned)q[1] + (unsigned)S.P.n[1] * (unsigned)q[2]);
    slot[w] = sh_ld16(L0.res + e * W);  // still the slots of cl_setup
    dg[w] = S.F.diag[pos];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const bool has_lo = q[d] > 0, has_hi = q[d] + 1 < S.P.n[d];
      const unsigned pl = has_lo ? lo_pos(S.P.n, q, pos, d) : pos, ph = has_hi ? hi_pos(S.P.n, q, pos, d) : pos;
      if (has_lo) T[w][2 * d] = S.F.T[d][pl];
      if (has_hi) T[w][2 * d + 1] = S.F.T[d][pos];
      na[w][2 * d] = cl_map(db + cl_local(L0, pl) * 8u, cl_owner(L0, pl));
      na[w][2 * d + 1] = cl_map(db + cl_local(L0, ph) * 8u, cl_owner(L0, ph));
    }
  }
  if (early) MDBS_PDL_WAIT();
  MDBS_PDL_TRIGGER();
#pragma unroll
  for (int w = 0; w < ROWS; w++)
    if (in[w]) {
      bc[w] = S.F.b[cl_position(L0, c.rank, w * kClThreads + t)];
      p[w] = S.F.p[nat[w]];
    }
  auto sync_all = [&] {
    if (ctas > 1) {
      cl_arrive();
      cl_wait();
    } else {
      __syncthreads();
    }
  };
  auto publish = [&](const double* v) {  // v of every cell to the exchanged vector
#pragma unroll
    for (int w = 0; w < ROWS; w++) sh_st(db + (w * kClRow + t) * 8u, v[w]);
    sync_all();
  };
  // (A v) at this thread's cell of row w
  auto apply = [&](int w, double own) {
    double xn[6];
#pragma unroll
    for (int d = 0; d < 6; d++)
      if (d < ne) cl_ld(na[w][d], xn[d]);
    double v = dg[w] * own;
#pragma unroll
    for (int d = 0; d < 6; d++)
      if (d < ne) v = fma(-T[w][d], xn[d], v);
    return v;
  };
  int par = 0;
  // The products' column chains and the trees over 32 columns, to every CTA: factors f[0]
  // f[1] and, with two sums, f[1] f[2] (squares: f[0] f[0] and f[1] f[1]); the two sums in
  // different warps.  One cluster barrier, which also separates the phases on either side.
  auto exchange = [&](const double (*f)[ROWS], int two, bool squares) {
    if (solo0) {  // a thread's cells are its column
      double a = 0.0, b = 0.0;
#pragma unroll
      for (int w = 0; w < ROWS; w++) {
        a = fma(f[0][w], f[squares ? 0 : 1][w], a);
        if (two) b = fma(f[1][w], f[squares ? 1 : kFactors - 1][w], b);
      }
      a = block_sum(a);
      if (two) b = block_sum(b);
      if (c.rank == 0 && warp == 0) {
        a = __shfl_sync(0xffffffffu, a, 0);
        b = __shfl_sync(0xffffffffu, b, 0);
        if ((int)lane < ctas) {
          cl_st(cl_map(sh_addr(&s_part[par][0][0]), lane), a);
          if (two) cl_st(cl_map(sh_addr(&s_part[par][1][0]), lane), b);
        }
      }
    } else {
#pragma unroll
      for (int k = 0; k < kFactors; k++)
        if (k < (squares ? 1 : 2) + two)
#pragma unroll
          for (int w = 0; w < ROWS; w++) s_fac[k][w * kClThreads + t] = f[k][w];
      __syncthreads();
      const unsigned which = t / (kClThreads / 2), col = t % (kClThreads / 2);
      if (col < kCols && (int)which <= two) {
        const double* fa = s_fac[which];
        const double* fb = s_fac[squares ? which : which + 1];
        double s = 0.0;
#pragma unroll
        for (int r = 0; r < kRepBig; r++) s = fma(fa[r * kCols + col], fb[r * kCols + col], s);
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        s = __shfl_sync(0xffffffffu, s, 0);
        const unsigned at = c.rank * ROWS + col / 32;
        if ((int)lane < ctas) cl_st(cl_map(sh_addr(&s_part[par][which][at]), lane), s);
      }
    }
    sync_all();
  };
  // the trees over a partial sum's eight warps and over the partial sums (one warp)
  auto total = [&](int which) {
    double v = (int)lane < slots ? s_part[par][which][lane] : 0.0;
    for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    v += __shfl_down_sync(0xffffffffu, v, 8);
    return __shfl_sync(0xffffffffu, v, 0);
  };
  double rr = 0.0, bb = 0.0, it = 0.0, rz = 0.0, alpha = 0.0;
  double f[kFactors][ROWS] = {};
  publish(p);
#pragma unroll
  for (int w = 0; w < ROWS; w++) {
    r[w] = in[w] ? bc[w] - apply(w, p[w]) : 0.0;
    f[0][w] = r[w];
    f[1][w] = bc[w];
  }
  exchange(f, 1, true);
  rr = total(0);
  bb = total(1);
  par ^= 1;
  const double limit = tol * sqrt(bb);
  // sqrt(rr) <= limit without the root where the answer is clear of rounding
  const double lim2 = limit * limit, lim_lo = lim2 * (1.0 - 1e-14), lim_hi = lim2 * (1.0 + 1e-14);
  const bool safe = lim2 > 1e-280 && lim2 < 1e280;
  auto converged = [&](double v) {
    if (safe && v < lim_lo) return true;
    if (safe && v > lim_hi) return false;
    return sqrt(v) <= limit;
  };
  bool done = bb == 0.0 || converged(rr) || it >= (double)max_it || !(rr == rr);
  if (bb == 0.0)  // b = 0 has the solution p = 0 whatever the initial guess
    for (int w = 0; w < ROWS; w++) p[w] = 0.0;
  const unsigned b0 = L0.b, x0 = L0.x;
  while (!done) {
#pragma unroll
    for (int w = 0; w < ROWS; w++)
      if (in[w]) sh_st(b0 + slot[w] * W, (R)r[w]);
    __syncthreads();  // the V-cycle's threads take their cells by slot
    if (!solo0) cl_arrive();
    cl_vcycle(c, 0, nlev, nu1, nu2, cs);
    if (!solo0) cl_wait();
    double z[ROWS];
#pragma unroll
    for (int w = 0; w < ROWS; w++) {
      R v = R(0);
      if (in[w]) sh_ld(x0 + slot[w] * W, v);
      z[w] = (double)v;
      f[0][w] = r[w];
      f[1][w] = z[w];
      if (kFlex) f[kFactors - 1][w] = qval[w];
    }
    exchange(f, kFlex ? 1 : 0, false);
    if (warp == 0) {
      const double nrz = total(0), zq = kFlex ? total(1) : 0.0;
      double be = 0.0;
      if (it != 0.0) be = kFlex ? -alpha * zq / rz : nrz / rz;
      rz = nrz;
      if (lane == 0) s_scal[0] = be;
    }
    __syncthreads();
    par ^= 1;
    const double be = s_scal[0];
#pragma unroll
    for (int w = 0; w < ROWS; w++) dval[w] = !in[w] ? 0.0 : (it == 0.0 ? z[w] : fma(be, dval[w], z[w]));
    publish(dval);
#pragma unroll
    for (int w = 0; w < ROWS; w++) {
      qval[w] = in[w] ? apply(w, dval[w]) : 0.0;
      f[0][w] = dval[w];
      f[1][w] = qval[w];
    }
    exchange(f, 0, false);
    if (warp == 0) {
      alpha = rz / total(0);
      if (lane == 0) s_scal[1] = alpha;
    }
    __syncthreads();
    par ^= 1;
    const double al = s_scal[1];
#pragma unroll
    for (int w = 0; w < ROWS; w++) {
      p[w] = fma(al, dval[w], p[w]);
      r[w] = in[w] ? fma(-al, qval[w], r[w]) : 0.0;
      f[0][w] = r[w];
    }
    exchange(f, 0, true);
    it += 1.0;
    if (warp == 0) {
      rr = total(0);
      const bool stop = converged(rr) || it >= (double)max_it || !(rr == rr);
      if (lane == 0) s_scal[2] = stop ? 1.0 : 0.0;
    }
    __syncthreads();
    par ^= 1;
    done = s_scal[2] != 0.0;
  }
#pragma unroll
  for (int w = 0; w < ROWS; w++)
    if (in[w]) S.F.p[nat[w]] = p[w];
  if (c.rank == 0 && t == 0) {
    double* scal = G.scal;
    scal[kBB] = bb;
    scal[kRR] = rr;
    scal[kIt] = it;
    scal[kCond] = 0.0;
  }
  sync_all();  // no CTA leaves while another may read its shared memory
}
