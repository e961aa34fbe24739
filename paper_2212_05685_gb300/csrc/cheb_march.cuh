// Recursion steps: FP32, NS steps per launch, and FP64 and double-float, one (included by
// cheb_kernels.cu).
//
// One CTA runs NS consecutive Chebyshev steps of a tile: CB = 2 NV columns, tx
// sites of the lattice rows (the whole row where it fits: `full`) and the
// lattice rows [y0, y1).  Stage s = 0 .. NS-1 computes
//   V_{m+s+1} = 2h~ V_{m+s} - V_{m+s-1}
// with its own warps, one thread per (site, column pair), marching along y.
//
// What bounds a step: the 13-point stencil is 100 packed FMAs per site row and
// column pair.  Read point by point it is 18 16-byte loads of V and 26 of the
// entries from shared memory, about 98 cycles of the SM's one shared-memory
// pipe per warp against 200 of one of its four FMA pipes: shared memory held the
// one-step kernel at 43% of the FMA pipe, one CTA of 512 threads in lockstep
// rows met its latencies, and at 24 B per row-column a step of slabs above L2
// cannot pass the memory's copy rate.  So
// - a thread keeps the three rows of its three sites x-1, x, x+1 in registers
//   (the row loop is unrolled by three, the windows' roles rotate): six loads of
//   V a row, and the entries, stored in the order of their use, come as
//   thirteen 16-byte loads;
// - a producer warp keeps several rows of V_m, V_{m-1} and entries in flight by
//   TMA (a row takes 2 to 3 us to land) and the stages wait for rows, not for
//   one another's warps;
// - the moment sums have a warp of their own: in the march they cost registers
//   (spills) and 5 us a launch;
// - with NS = 2 the slabs are streamed once for two steps (32 instead of 48 B per
//   row-column), stage 0 handing its rows to stage 1 in shared memory, for
//   NS - 1 - s more sites and rows on each side of the tile recomputed by stage s.
//   A code copy per stage missed the instruction cache: the stages share one.
// The terms of a row's sum are those of stencil_site in the same order, so every
// number of the recursion has the same bits whatever NS, tile and band.
//
// Measured against the one-step kernel with block-shared windows, us per step:
// 37x29 40.0 -> 20.8 (18.3 where launches overlap), 48x24 31.8 -> 16.7 (one step, slabs in L2), 64x64 343 ->
// 266 (one step, 90% of the copy rate; 217 in parts that fit L2), 100x100 1655 -> 1248 (two steps; one
// step: 1457 = 97% of the copy rate), its eighth (2500 columns) 237 -> 180.
// FP64 and double-float elements (one complex number of 16 bytes in place of a column
// pair, 24 cmac and two real products a site) are bound by their arithmetic; the march
// keeps its warps out of row lockstep: FP64 16x16, M = 256, 9.45 -> 7.14 ms (6.5 at the
// FP64 rate), double-float 48x24, M = 1024, 165.7 -> 160.8, and with packed arithmetic 113.7
// (about 85 at the FP32 rate).
//
// Rings and barriers (indices count rows of a stage from its first row).
// Set i = {V_m row i + 2 (set 0: rows 0, 1, 2), V_{m-1} row i, entries row i}
// lands on full[i]; the warps of stage s and the warp of the sums arrive on
// done_s[i] when they have finished row i.  Stage s at row i reads input row
// i + 2 (at i = 0 rows 0 .. 2), entries row i + s, and as subtrahend V_{m-1} row i
// or, s > 0, row i + 2 of stage s - 1's input; the sums read input rows i .. i + 2.
// A set is issued once the last stage has finished row i - lag, so stage s row
// i - lag + 2 (NS - 1 - s); the ring sizes follow (plan_march) and a test replays
// them.  Every wait is bounded: a CTA whose waits run out writes
// NaN over the rows and columns it owns.

// elements: FP32 column pairs, double-float and FP64 complex numbers, 16 bytes each
enum { kElF32 = 0, kElDF = 1, kElF64 = 2 };
constexpr int kMarchLanes = 8;      // elements of a Nambu row per CTA
constexpr int march_cols(int el) { return el == kElF32 ? 2 * kMarchLanes : kMarchLanes; }
constexpr int march_entry_bytes(int el) { return el == kElF32 ? 208 : 400; }  // of a site (13, 25 times 16)
constexpr int kMarchThreads = 512;  // 16 warps: 128 registers a thread for the 3 x 3 x 2 window and two sums
// what two slabs touch stays in L2 (129 MB) up to this size: 48x24 (85 MB) runs a step in
// 16.7 us one step per launch, in 25.3 us two, where the halo sites and rows only cost
constexpr int64_t kMarchL2 = 100000000;
constexpr int kMarchBars = 16;      // phases of every barrier ring
constexpr int kMarchRows = 8;       // rows of every ring of a launch of several steps

// boxes of a slab's rows: a tile with the sites around it, with those of one side,
// and the sites of the other side (full rows: mid only)
struct MarchMaps {
  CUtensorMap mid, edge, halo;
};

struct MarchArgs {
  int nx, ny;
  int64_t D, ldq;
  int tx, ntile, full, ylen;
  int wrow;             // sites of a ring row: the tile's and ns more on each side (full: nx)
  int lag;              // a set is issued once the last stage has finished the row `lag` before it
  int rp, rv, rs, rc;   // rows of the rings: V_{m-1}, V_m, between stages, entries
  int rowb;             // bytes of a ring row of vectors
  int crowb;            // bytes of a row of entries (a multiple of 128, in memory and in the ring)
  const float4* table;  // [ny][ntile][wrow][13]: the entries of a ring row's sites in the order of their use
  float4 *outa, *outb;  // V_{m+NS-1} (NS > 1) and V_{m+NS}
  double2* acc;
  const double* am;
  const double* ao;
  int m;
  int chunk0;           // the launch's first column chunk
  int64_t grow;         // bytes of a lattice row of a slab
};

__device__ __forceinline__ uint32_t mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred q;\n elect.sync _|q, 0xffffffff;\n selp.u32 %0, 1, 0, q;\n}\n" : "=r"(p));
  return p != 0;
}

template <int NV>
struct MarchRow {  // sites x-1, x, x+1 of a row: e = the thread's first component, h = the other
  ulonglong2 e[3], h[3];
};

// wait of a march warp: the fast path is one poll; the slow path gives up at the
// limit or as soon as another warp of the CTA has
__device__ __forceinline__ bool march_wait_slow(uint32_t bar, uint32_t parity, uint64_t limit_ns, volatile int* fail) {
  const uint64_t t0 = global_ns();
#pragma unroll 1
  for (uint32_t it = 1; it < (1u << 26); ++it) {
    if (mbar_try(bar, parity)) return true;
    if ((it & 63) == 0 && (*fail != 0 || global_ns() - t0 > limit_ns)) return false;
  }
  return false;
}

// one row of one component of the thread's site: P = sum Re(c) v, Q = sum Im(c) v in the
// term order of stencil_site (diagonal, then the neighbours (+1,0) (-1,0) (0,+1)
// (0,-1) (+1,+1) (-1,-1) (+1,-1) (-1,+1)); C = 0, 1: the component read first, the other.
// The two components one after the other: half the sums live at a time.
template <int NV, int C>
__device__ __forceinline__ ulonglong2 march_stencil(const MarchRow<NV>& wm, const MarchRow<NV>& w0,
                                                    const MarchRow<NV>& wp, const float4* cq, float4& q) {
  Acc2 a = {0ull, 0ull, 0ull, 0ull};
  constexpr int I0 = 25 * C;
  auto entry = [&](int i) {  // stored float i, read in order
    if ((i & 3) == 0) q = cq[i >> 2];
    return (i & 3) == 0 ? q.x : (i & 3) == 1 ? q.y : (i & 3) == 2 ? q.z : q.w;
  };
  auto own = [&](const MarchRow<NV>& w, int d) { return C ? w.h[d] : w.e[d]; };
  auto oth = [&](const MarchRow<NV>& w, int d) { return C ? w.e[d] : w.h[d]; };
  {
    const u64 d = dup2(entry(I0));
    const ulonglong2 u = own(w0, 1);
    a.pr = f2fma(d, u.x, a.pr);
    a.pi = f2fma(d, u.y, a.pi);
  }
  auto term = [&](int k, const MarchRow<NV>& w, int d) {
    const int i = I0 + (k < 4 ? 1 + 4 * k : 17 + 2 * (k - 4));
    float re = entry(i), im = entry(i + 1);
    acc_term(a, make_float2(re, im), own(w, d));
    if (k < 4) {
      re = entry(i + 2);
      im = entry(i + 3);
      acc_term(a, make_float2(re, im), oth(w, d));
    }
  };
  term(0, w0, 2);
  term(1, w0, 0);
  term(2, wp, 1);
  term(3, wm, 1);
  term(4, wp, 2);
  term(5, wm, 0);
  term(6, wm, 2);
  term(7, wp, 0);
  return make_ulonglong2(f2sub(a.pr, a.qi), f2add(a.pi, a.qr));
}

// the same for one complex number per element, starting from minus `b` (FIRST: from
// nothing, and halved); a site's entries are its two real diagonals (one element), then
// per component twelve of 16 bytes.  FP64: the operations of cmac.
template <int NV, int C, bool FIRST>
__device__ __forceinline__ ulonglong2 march_stencil_f64(const MarchRow<NV>& wm, const MarchRow<NV>& w0,
                                                        const MarchRow<NV>& wp, const double2* cq, ulonglong2 b) {
  auto el = [](ulonglong2 u) { return make_double2(__longlong_as_double((long long)u.x), __longlong_as_double((long long)u.y)); };
  auto own = [&](const MarchRow<NV>& w, int d) { return el(C ? w.h[d] : w.e[d]); };
  auto oth = [&](const MarchRow<NV>& w, int d) { return el(C ? w.e[d] : w.h[d]); };
  double2 a = FIRST ? make_double2(0.0, 0.0) : vneg(el(b));
  rmac(a, C ? cq[0].y : cq[0].x, own(w0, 1));
  const double2* c = cq + 1 + 12 * C;
  auto term = [&](int k, const MarchRow<NV>& w, int d) {
    const int i = k < 4 ? 2 * k : 8 + (k - 4);
    cmac(a, c[i], own(w, d));
    if (k < 4) cmac(a, c[i + 1], oth(w, d));
  };
  term(0, w0, 2);
  term(1, w0, 0);
  term(2, wp, 1);
  term(3, wm, 1);
  term(4, wp, 2);
  term(5, wm, 0);
  term(6, wm, 2);
  term(7, wp, 0);
  if (FIRST) a = vhalf(a);
  return make_ulonglong2((u64)__double_as_longlong(a.x), (u64)__double_as_longlong(a.y));
}

// Double-float: an element is (re_hi, im_hi), (re_lo, im_lo), and every operation
// of df_mac works on both parts at once, which halves the instructions issued: the scalar
// form is 1200 of them a site, 71% of the issue slots and 56% of the FMA pipe.  The
// products with the real and with the imaginary part of an entry are summed apart, P and
// Q as in FP32 (no part of v changes place), and joined at the end.
__device__ __forceinline__ void df_mac2(ulonglong2& a, float ch, float cl, ulonglong2 v) {
  const u64 h = dup2(ch);
  const u64 np = f2mul(dup2(-ch), v.x);  // minus the product
  u64 e = f2fma(h, v.x, np);
  e = f2fma(h, v.y, e);
  e = f2fma(dup2(cl), v.x, e);
  const u64 s = f2sub(a.x, np);
  const u64 bb = f2sub(s, a.x);
  const u64 t = f2sub(f2sub(a.x, f2sub(s, bb)), f2add(np, bb));
  a.x = s;
  a.y = f2add(a.y, f2add(t, e));
}
// two_sum of both parts
__device__ __forceinline__ void two_sum2(u64 a, u64 b, u64& s, u64& e) {
  s = f2add(a, b);
  const u64 bb = f2sub(s, a);
  e = f2add(f2sub(a, f2sub(s, bb)), f2sub(b, bb));
}
template <int NV, int C, bool FIRST>
__device__ __forceinline__ ulonglong2 march_stencil_df(const MarchRow<NV>& wm, const MarchRow<NV>& w0,
                                                       const MarchRow<NV>& wp, const float4* cq, ulonglong2 b) {
  auto own = [&](const MarchRow<NV>& w, int d) { return C ? w.h[d] : w.e[d]; };
  auto oth = [&](const MarchRow<NV>& w, int d) { return C ? w.e[d] : w.h[d]; };
  constexpr u64 kSigns = 0x8000000080000000ull;
  ulonglong2 P = FIRST ? make_ulonglong2(0ull, 0ull) : make_ulonglong2(b.x ^ kSigns, b.y ^ kSigns);
  ulonglong2 Q = make_ulonglong2(0ull, 0ull);
  {
    const float4 d = cq[0];
    df_mac2(P, C ? d.z : d.x, C ? d.w : d.y, own(w0, 1));
  }
  const float4* c = cq + 1 + 12 * C;
  auto mac = [&](float4 e, ulonglong2 v) {
    df_mac2(P, e.x, e.y, v);
    df_mac2(Q, e.z, e.w, v);
  };
  auto term = [&](int k, const MarchRow<NV>& w, int d) {
    const int i = k < 4 ? 2 * k : 8 + (k - 4);
    mac(c[i], own(w, d));
    if (k < 4) mac(c[i + 1], oth(w, d));
  };
  term(0, w0, 2);
  term(1, w0, 0);
  term(2, wp, 1);
  term(3, wm, 1);
  term(4, wp, 2);
  term(5, wm, 0);
  term(6, wm, 2);
  term(7, wp, 0);
  // P + i Q, once renormalised
  const u64 qh = ((Q.x >> 32) | (Q.x << 32)) ^ 0x80000000ull, ql = ((Q.y >> 32) | (Q.y << 32)) ^ 0x80000000ull;
  u64 h, t;
  two_sum2(P.x, qh, h, t);
  u64 l = f2add(f2add(P.y, ql), t);
  if (FIRST) {
    const u64 half2 = 0x3F0000003F000000ull;  // (0.5f, 0.5f)
    h = f2mul(h, half2);
    l = f2mul(l, half2);
  }
  ulonglong2 o;
  two_sum2(h, l, o.x, o.y);
  return o;
}

// where site k of a tile of w <= tx sites sits in a ring row: after the ns sites on its
// left; the sites on its right follow the full tile's
__device__ __forceinline__ int march_pos(int k, int w, int tx, int ns) { return k < w ? ns + k : ns + tx + (k - w); }
// byte offset in a ring row of what slot s of column c of a chunk (own component
// beta) reads, its site at position p; and its value in FP64
template <int EL, int NV>
__device__ __forceinline__ int march_item(int p, int s, int beta, int c) {
  return p * 32 * NV + (beta ^ kSlotFlip[s]) * 16 * NV + (EL == kElF32 ? (c >> 1) * 16 + (c & 1) * 4 : c * 16);
}
template <int EL>
__device__ __forceinline__ double2 march_value(const unsigned char* at) {
  if (EL == kElF64) return *reinterpret_cast<const double2*>(at);
  const float* e = reinterpret_cast<const float*>(at);
  if (EL == kElF32) return make_double2((double)e[0], (double)e[2]);
  return make_double2((double)e[0] + (double)e[2], (double)e[1] + (double)e[3]);
}

template <int EL, int NS, bool FIRST, bool HOOK>
__global__ void __launch_bounds__(kMarchThreads, 1)
    cheb_march_kernel(const __grid_constant__ MarchMaps vm, const __grid_constant__ MarchMaps pm,
                      const __grid_constant__ MarchArgs a, const __grid_constant__ ColMap cmap) {
  constexpr int NV = kMarchLanes;
  constexpr int COLS = march_cols(EL), ENTRYB = march_entry_bytes(EL);
  constexpr int SITE = 2 * NV;         // float4 per site of a row
  constexpr int SITEB = 16 * SITE;     // bytes
  constexpr int LAST = NS - 1;
  const int nx = a.nx, ny = a.ny;
  const bool full = a.full != 0;

  extern __shared__ __align__(1024) unsigned char smem_march[];
  // from its start: the rings of V_{m-1}, of V_m and between the stages, the ring of the
  // entries, barriers.  Every ring row holds the same sites.
  const int rowb = a.rowb, crowb = a.crowb;
  const int vbase = a.rp * rowb, sbase = vbase + a.rv * rowb, sring = a.rs * rowb;
  const int cbase = sbase + LAST * sring;
  const int bbase = cbase + a.rc * crowb;
  uint64_t* const bars = reinterpret_cast<uint64_t*>(smem_march + bbase);
  volatile int* const fail = reinterpret_cast<volatile int*>(bars + kMarchBars * (1 + NS));

  const int tile = blockIdx.x % a.ntile;
  const int y0 = (blockIdx.x / a.ntile) * a.ylen;
  const int nrow = min(ny, y0 + a.ylen) - y0;
  const int x0 = tile * a.tx;
  const int w = min(nx, x0 + a.tx) - x0;
  const int64_t cb0 = (int64_t)(a.chunk0 + blockIdx.y) * COLS;
  const int64_t q0 = (int64_t)(a.chunk0 + blockIdx.y) * NV;
  const int nset = nrow + 2 * LAST;  // rows of stage 0

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  // warps of stage s: the launch has them for a full tile's width
  int first_warp[NS + 1];
  first_warp[0] = 0;
#pragma unroll
  for (int s = 0; s < NS; ++s)
    first_warp[s + 1] = first_warp[s] + ((full ? nx : a.tx + 2 * (LAST - s)) * NV + 31) / 32;

  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int i) { return bar0 + 8 * (i & (kMarchBars - 1)); };
  auto done_bar = [&](int s, int i) { return bar0 + 8 * (kMarchBars * (1 + s) + (i & (kMarchBars - 1))); };
  auto parity = [](int i) { return (uint32_t)((i / kMarchBars) & 1); };
  auto limit = [&]() -> uint64_t {
    return HOOK ? (uint64_t)*reinterpret_cast<volatile unsigned long long*>(&g_wait_limit_ns) : kWaitLimitNs;
  };
  // warp-wide wait: the same answer on every lane
  auto wait = [&](uint32_t bar, int i) {
    if (__all_sync(0xffffffffu, mbar_try(bar, parity(i)))) return true;
    return __all_sync(0xffffffffu, march_wait_slow(bar, parity(i), limit(), fail)) != 0;
  };

  // launched programmatically, a CTA starts while the launch before finishes: it touches
  // no slab, sum or entry before this
  auto grid_wait = [&]() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); };
  auto poison = [&]() {  // NaN over the tile's outputs
    grid_wait();
    const float nan = __int_as_float(-1);  // all bits set: NaN as FP32 and, two of them, as FP64
    const float4 nan4 = make_float4(nan, nan, nan, nan);
    for (int t = threadIdx.x; t < nrow * 2 * w * NV; t += blockDim.x) {
      const int r = t / (2 * w * NV), k = t - r * (2 * w * NV);
      const int64_t g = (2 * ((int64_t)(y0 + r) * nx + x0) + k / NV) * a.ldq + q0 + k % NV;
      if (NS > 1) a.outa[g] = nan4;
      a.outb[g] = nan4;
    }
  };
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
  // after a fault anywhere, later CTAs and launches only mark their outputs
  if (*reinterpret_cast<volatile unsigned int*>(&g_step_fault) != 0u) {
    poison();
    return;
  }
  const bool aligned = (smem_u32(smem_march) & 127u) == 0;
  if (aligned && threadIdx.x == 0) {
    for (int k = 0; k < kMarchBars; ++k) mbar_init(bar0 + 8 * k, 1);
    for (int s = 0; s < NS; ++s)
      for (int k = 0; k < kMarchBars; ++k) mbar_init(done_bar(s, k), first_warp[s + 1] - first_warp[s] + 1);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  }
  if (!__syncthreads_and(aligned)) {
    if (threadIdx.x == 0) atomicOr(&g_step_fault, 2u);
    poison();
    return;
  }

  grid_wait();

  if (warp == first_warp[NS]) {
    // producer: the sets, as soon as the ring rows they overwrite are free.  The whole
    // warp runs the loop (so that ring positions, rows and waits stay in the uniform
    // datapath); one elected lane issues
    const uint32_t p0 = smem_u32(smem_march), v0 = p0 + vbase, c0 = p0 + cbase;
    const uint32_t vend = p0 + sbase, pend = p0 + vbase, cend = p0 + bbase;
    const uint32_t bytes = rowb + crowb + (FIRST ? 0u : (uint32_t)(full ? nx : a.tx + 2 * LAST) * SITEB);
    const int col = (int)(4 * q0), nx2 = 2 * nx;
    // a tile's row with the sites around it is one box, or two where it wraps around
    // the lattice: edge = 0 no (or the whole row), 1 on the left, 2 on the right
    const int edge = full ? 0 : x0 == 0 ? 1 : x0 + w == nx ? 2 : 0;
    const int vrow = full || edge == 1 ? 2 * x0 : 2 * (x0 - NS), vhrow = edge == 1 ? 2 * (nx - NS) : 0;
    const int prow = full || edge == 1 ? 2 * x0 : 2 * (x0 - LAST), phrow = edge == 1 ? 2 * (nx - LAST) : 0;
    const int vdst = edge == 1 ? NS * SITEB : 0, vhdst = edge == 1 ? 0 : (NS + a.tx) * SITEB;
    const int pdst = full ? 0 : edge == 1 ? NS * SITEB : SITEB, phdst = edge == 1 ? SITEB : (NS + a.tx) * SITEB;
    uint32_t vd = v0, pd = p0, cd = c0;
    int yv = wrapi(y0 - LAST - 1, ny), yc = wrapi(y0 - LAST, ny);  // lattice rows of the next V_m row, of set i
    const int cstep = a.ntile * (crowb / 16);  // float4 of a lattice row of entries, tile by tile
    const float4* const ctile = a.table + tile * (crowb / 16);
    const float4* csrc = ctile + (int64_t)yc * cstep;
    const bool leader = elect_one();
    bool ok = true;
    int issued = -1;
    auto load_v = [&](uint32_t bar, bool skip) {
      const int row = nx2 * yv;
      if (leader && !skip) {
        if (edge == 0) {
          tma_load_2d(vd, &vm.mid, col, row + vrow, bar);
        } else {
          tma_load_2d(vd + vdst, &vm.edge, col, row + vrow, bar);
          tma_load_2d(vd + vhdst, &vm.halo, col, row + vhrow, bar);
        }
      }
      vd = vd + rowb == vend ? v0 : vd + rowb;
      yv = yv + 1 == ny ? 0 : yv + 1;
    };
    // test hook: the third window row of set 0 is skipped, so its phase stays open
    bool skip = false;
    if (HOOK) {
      if (leader) skip = *reinterpret_cast<volatile int*>(&g_drop_copy) > 0 && atomicSub(&g_drop_copy, 1) > 0;
    }
    if (leader) mbar_expect_tx(full_bar(0), bytes + 2 * rowb);
    load_v(full_bar(0), false);
    load_v(full_bar(0), false);
#pragma unroll 1
    for (int i = 0; i < nset; ++i) {
      // the ring rows that the set overwrites have been read once the last stage has
      // finished row i - lag (the ring sizes follow from that, plan_march); before its
      // first rows, once a stage before it has finished the rows it leads by
      int st = LAST, r = i - a.lag;
      while (r < 0 && st > 0) {
        r += 2;
        --st;
      }
      if (r >= 0) ok = wait(done_bar(st, r), r);
      if (!ok) break;
      const uint32_t bar = full_bar(i);
      if (leader && i > 0) mbar_expect_tx(bar, bytes);
      load_v(bar, HOOK && i == 0 && skip);
      const int row = nx2 * yc;
      if (leader) {
        if (!FIRST) {
          if (LAST == 0 || edge == 0) {
            tma_load_2d(pd + pdst, &pm.mid, col, row + prow, bar);
          } else {
            tma_load_2d(pd + pdst, &pm.edge, col, row + prow, bar);
            tma_load_2d(pd + phdst, &pm.halo, col, row + phrow, bar);
          }
        }
        bulk_load(cd, csrc, crowb, bar);
      }
      pd = pd + rowb == pend ? p0 : pd + rowb;
      cd = cd + crowb == cend ? c0 : cd + crowb;
      ++yc;
      csrc += cstep;
      if (yc == ny) {
        yc = 0;
        csrc = ctile;
      }
      issued = i;
    }
    if (!ok && lane == 0) *fail = 1;
    __syncwarp();
    if (*fail && lane == 0)  // copies may still be in flight: wait (bounded) for every phase armed last
      for (int i = max(0, issued - kMarchBars + 1); i <= issued; ++i)
        mbar_wait_slow(full_bar(i), parity(i), limit() >> 2);
  } else if (warp == first_warp[NS] + 1) {
    // moment sums a_{m+s} V_{m+s} of every stage's input, by a warp of their own (in the
    // march they cost its registers, and a lone thread's twenty FP64 sums 5 us a
    // launch): row by row it waits for the stage's input rows, adds the sums of the
    // chunk's columns whose own site lies in the row and the tile, and arrives beside the stage's warps, which holds the rows it reads
    const bool sums = a.acc != nullptr;
    // unit columns: lane + 32 k is slot (lane + 32 k) % 10 of column (lane + 32 k) / 10
    constexpr int ITEMS = (COLS * kSlots + 31) / 32;
    int iy[ITEMS], off[ITEMS];
    if (sums) {
#pragma unroll
      for (int q = 0; q < ITEMS; ++q) {
        const int t = lane + 32 * q, c = t / kSlots, sl = t - c * kSlots;
        const int64_t col = cmap.s0 + cb0 + c;
        iy[q] = -1;
        off[q] = 0;
        if (c < COLS && col < (a.D >> cmap.js)) {
          const int J = (int)(col << cmap.js), j = J >> 1;
          const int xj = j % nx, k = xj - x0;
          if (k >= 0 && k < w) iy[q] = j / nx;
          off[q] = march_item<EL, NV>(full ? wrapi(xj + kSlotDx[sl], nx) : march_pos(k + kSlotDx[sl], w, a.tx, NS), sl,
                                  J & 1, c);
        }
      }
    }
    // lattice rows with sums of the chunk: none but those take more than the wait and the arrival
    int ylo = ny, yhi = -1;
    double cms[NS], cos[NS];
    if (sums) {
      const int64_t c0 = cmap.s0 + cb0, c1 = min(a.D >> cmap.js, c0 + COLS) - 1;
      if (c1 >= c0) {
        ylo = (int)((c0 << cmap.js) >> 1) / nx;
        yhi = (int)((c1 << cmap.js) >> 1) / nx;
      }
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        cms[s] = a.am[a.m + s];
        cos[s] = a.ao[a.m + s];
      }
    }
    bool ok = true;
#pragma unroll 1
    for (int tt = 0; tt < nset && ok; ++tt) {
#pragma unroll
      for (int s = 0; s < NS && ok; ++s) {
        const int i = tt - 2 * s, G = LAST - s;
        if (i < 0 || i >= nrow + 2 * G) continue;
        ok = s == 0 ? wait(full_bar(i), i) : wait(done_bar(s > 0 ? s - 1 : 0, i + 2), i + 2);
        const int y = y0 + i - G;
        if (ok && i >= G && i < G + nrow && y >= ylo && y <= yhi && !(FIRST && s == 0)) {
          const double cm = cms[s], co = cos[s];
          // ring rows of y - 1, y, y + 1
          const int rbase = s == 0 ? vbase : sbase + (s - 1) * sring, rows = s == 0 ? a.rv : a.rs;
          int rowat[3];
#pragma unroll
          for (int d = 0; d < 3; ++d) rowat[d] = rbase + (i + d) % rows * rowb;
          double2 old[ITEMS];
#pragma unroll
          for (int q = 0; q < ITEMS; ++q) {
            const int t = lane + 32 * q;
            if (iy[q] == y) old[q] = a.acc[((cmap.s0 + cb0 + t / kSlots) << cmap.js) * kSlots + t % kSlots];
          }
#pragma unroll
          for (int q = 0; q < ITEMS; ++q) {
            if (iy[q] != y) continue;
            const int t = lane + 32 * q, sl = t % kSlots;
            const int64_t J = (cmap.s0 + cb0 + t / kSlots) << cmap.js;
            const double2 e = march_value<EL>(
                smem_march + (kSlotDy[sl] < 0 ? rowat[0] : kSlotDy[sl] > 0 ? rowat[2] : rowat[1]) + off[q]);
            acc_add_unit(&old[q], sl == kSlots - 1 ? co : cm, e.x, e.y);
            a.acc[J * kSlots + sl] = old[q];
            if (sl == 0 && cmap.rec) record_diag(cmap, a.D, a.m + s, J, make_double2(1.0, 0.0), e.x, e.y);
          }
        }
        __syncwarp();
        if (ok && lane == 0) mbar_arrive(done_bar(s, i));
      }
    }
    if (!ok && lane == 0) *fail = 1;
  } else {
    // the march of stage st over its rows: one code for every stage, so that all
    // warps run the same instructions (a copy per stage missed the instruction cache)
    int st = 0;
#pragma unroll
    for (int s = 1; s < NS; ++s)
      if (warp >= first_warp[s]) st = s;
    const int G = LAST - st;  // sites and rows beyond the tile on each side
    const int nrows = nrow + 2 * G;
    int fw = 0;
#pragma unroll
    for (int s = 1; s < NS; ++s)
      if (st == s) fw = first_warp[s];
    const int t = threadIdx.x - 32 * fw;
    const int v = t % NV;
    const int lx = t / NV;
    const bool on = full ? lx < nx : lx < w + 2 * G;
    const int k = on ? (full ? lx : lx - G) : 0;  // site x0 + k of the lattice row (wrapped)
    const int x = full ? k : wrapi(x0 + k, nx);
    const bool own = on && (full || (k >= 0 && k < w));
    constexpr int hd = 16 * NV;  // the site's other component
    // where site k of the tile sits in a ring row: after the ns sites on its left; the
    // sites on its right follow the full tile's
    auto pos = [&](int kk) {
      return full ? (kk < 0 ? kk + nx : (kk >= nx ? kk - nx : kk)) : march_pos(kk, w, a.tx, NS);
    };
    // the thread's sites x - 1, x, x + 1 in a ring row, its entries
    const int off0 = pos(k - 1) * SITEB + 16 * v, off1 = pos(k) * SITEB + 16 * v, off2 = pos(k + 1) * SITEB + 16 * v;
    const int ocf = pos(k) * ENTRYB;
    // running positions in the rings of the input, the subtrahend, the output, the entries
    const int inb = st == 0 ? vbase : sbase + (st - 1) * sring, ine = st == 0 ? sbase : inb + sring;
    const int pvb = st == 0 ? 0 : st == 1 ? vbase : sbase + (st - 2) * sring;
    const int pve = st == 0 ? vbase : st == 1 ? sbase : pvb + sring;
    const int sob = sbase + st * sring;
    // (several steps: eight rows each, so that positions follow from the row's index)
    int oi = inb + 2 * rowb, op = pvb, oo = sob, oc = cbase;
    char* gp = reinterpret_cast<char*>(st == LAST ? a.outb : a.outa) +
               16 * (2 * ((int64_t)y0 * nx + x) * a.ldq + q0 + v);

    MarchRow<NV> wa, wb, wc;
    auto ld16 = [&](int off) { return *reinterpret_cast<const ulonglong2*>(smem_march + off); };
    auto load_row = [&](MarchRow<NV>& r, int base) {
      r.e[0] = ld16(base + off0);
      r.h[0] = ld16(base + off0 + hd);
      r.e[1] = ld16(base + off1);
      r.h[1] = ld16(base + off1 + hd);
      r.e[2] = ld16(base + off2);
      r.h[2] = ld16(base + off2 + hd);
    };
    // barriers of row i's input and of the ring row it overwrites, and their rows
    const bool from_ring = NS > 1 && st > 0;
    auto in_row = [&](int i) { return from_ring ? i + 2 : i; };
    auto in_bar = [&](int i) { return from_ring ? done_bar(st - 1, i + 2) : full_bar(i); };
    auto out_two = [&](int i) { return st + 2 <= LAST && i >= kMarchRows + 2; };
    auto out_row = [&](int i) { return out_two(i) ? i - kMarchRows - 2 : i - kMarchRows; };
    auto out_bar = [&](int i) { return done_bar(out_two(i) ? st + 2 : st + 1, out_row(i)); };
    bool ready = false;

    auto row = [&](int i, const MarchRow<NV>& rm, const MarchRow<NV>& r0, MarchRow<NV>& rp) -> bool {
      // the input row (and with it the entries: the stage before has read row i + st of
      // them), and the ring row this row overwrites: read by stage st + 1, its moment
      // sums and, as subtrahend, by stage st + 2.  (The single step tests the next row's
      // barrier a row ahead, so that its latency is not met between the rows.)
      if (!ready) {
        if (!wait(in_bar(i), in_row(i))) return false;
        if (NS > 1 && st < LAST && i >= kMarchRows && !wait(out_bar(i), out_row(i))) return false;
      }
      uint32_t next = 0;
      if (NS == 1) next = mbar_test(in_bar(i + 1), parity(i + 1));
      if (NS > 1) {
        oi = inb + ((i + 2) & (kMarchRows - 1)) * rowb;
        op = pvb + ((st > 0 ? i + 2 : i) & (kMarchRows - 1)) * rowb;
        oo = sob + (i & (kMarchRows - 1)) * rowb;
        oc = cbase + ((i + st) & (kMarchRows - 1)) * crowb;
      }
      load_row(rp, oi);
      const float4* cq = reinterpret_cast<const float4*>(smem_march + ocf + oc);
      const int p = op + off1;
      if (NS == 1) {
        oi = oi + rowb == ine ? inb : oi + rowb;
        op = op + rowb == pve ? pvb : op + rowb;
        oc = oc + crowb == bbase ? cbase : oc + crowb;
      }
      ulonglong2 o0, o1;
      if constexpr (EL == kElF32) {
        float4 q;
        o0 = march_stencil<NV, 0>(rm, r0, rp, cq, q);
        o1 = march_stencil<NV, 1>(rm, r0, rp, cq, q);
        if (FIRST && st == 0) {
          const u64 half2 = 0x3F0000003F000000ull;  // (0.5f, 0.5f)
          o0.x = f2mul(o0.x, half2);
          o0.y = f2mul(o0.y, half2);
          o1.x = f2mul(o1.x, half2);
          o1.y = f2mul(o1.y, half2);
        } else {
          const ulonglong2 b0 = ld16(p), b1 = ld16(p + hd);
          o0.x = f2sub(o0.x, b0.x);
          o0.y = f2sub(o0.y, b0.y);
          o1.x = f2sub(o1.x, b1.x);
          o1.y = f2sub(o1.y, b1.y);
        }
      } else {
        const ulonglong2 b0 = FIRST ? make_ulonglong2(0ull, 0ull) : ld16(p), b1 = FIRST ? b0 : ld16(p + hd);
        if constexpr (EL == kElDF) {
          o0 = march_stencil_df<NV, 0, FIRST>(rm, r0, rp, cq, b0);
          o1 = march_stencil_df<NV, 1, FIRST>(rm, r0, rp, cq, b1);
        } else {
          const double2* cd = reinterpret_cast<const double2*>(cq);
          o0 = march_stencil_f64<NV, 0, FIRST>(rm, r0, rp, cd, b0);
          o1 = march_stencil_f64<NV, 1, FIRST>(rm, r0, rp, cd, b1);
        }
      }
      if (NS > 1 && st < LAST) {
        if (on) {
          unsigned char* r = smem_march + off1 + oo;
          *reinterpret_cast<ulonglong2*>(r) = o0;
          *reinterpret_cast<ulonglong2*>(r + hd) = o1;
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(done_bar(st, i));
      // (after the arrival: nobody in the CTA waits for the stores)
      if (i >= G && i < G + nrow) {
        if (own && (NS < 3 || st >= NS - 2)) {
          *reinterpret_cast<ulonglong2*>(gp) = o0;
          *reinterpret_cast<ulonglong2*>(gp + 16 * a.ldq) = o1;
        }
        gp += a.grow;
      }
      if (NS == 1) ready = __all_sync(0xffffffffu, next != 0);
      return true;
    };

    // rows 0 and 1 of the input, then the rows with the window's three rows in turn
    bool ok = st == 0 ? wait(full_bar(0), 0) : wait(done_bar(NS > 1 && st > 0 ? st - 1 : 0, 1), 1);
    if (ok) {
      load_row(wa, inb);
      load_row(wb, inb + rowb);
#pragma unroll 1
      for (int i = 0; i < nrows; i += 3) {
        if (!(ok = row(i, wa, wb, wc))) break;
        if (i + 1 < nrows && !(ok = row(i + 1, wb, wc, wa))) break;
        if (i + 2 < nrows && !(ok = row(i + 2, wc, wa, wb))) break;
      }
    }
    if (!ok && lane == 0) *fail = 1;
  }
  __syncthreads();
  if (*fail) {
    if (threadIdx.x == 0) atomicOr(&g_step_fault, 1u);
    poison();
  }
}
