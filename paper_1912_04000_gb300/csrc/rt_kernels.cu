// Wavefront path-tracing kernels (sm_103a).
//
// One wave holds up to C spectral paths (view, pixel, sample, band).  For each
// vertex k = 1..depth the host enqueues three kernels:
//   k_trace4 - closest hit of every queued ray over the four-wide BVH (k_trace:
//              the binary, eight-wide and 8-bit-quantised trees, options;
//              watertight FP32 test), persistent warps refilling idle lanes
//              from the queue, leaf batching;
//   k_shade  - material event at the hit (section 4: Eq. 2 by cosine sampling
//              for stone, thin-glass/conductor Fresnel events with the complex
//              index of Eq. 1), next-event estimate of the sun cone (Eq. 3),
//              continuation ray appended to the next queue;
//   k_shadow4 - transmittance of the sun rays (0 behind stone, product of the
//              thin-glass T_s otherwise), added to the path's radiance
//              (k_shadow: over the binary BVH).
// The FP64 accumulation into the spectral image needs no atomics: in a wave of
// one sample or less each path owns its output slot (pixel, band), and waves
// run in sample order; in a wave of several samples paths leave their radiance
// in the wave and k_resolve adds it up per slot, in sample order.
#include <algorithm>
#include <cstdio>
#include <type_traits>

#include "rt_device.cuh"

namespace srt {

namespace {

// ---------------------------------------------------------------------------
// BVH traversal as a resumable per-lane state machine.  One call of a step
// function visits one interior node (both children tested, the far one
// pushed) or one leaf, then pops if needed; it returns true when the ray is
// finished.  The persistent kernels below interleave steps with refills of
// idle lanes, so a warp never waits for its longest ray with most lanes idle.
//
// FMA selects the box test: false = (plane - o) * inv (any origin); true =
// fma(plane, inv, -o * inv), valid for origins within the scene bounds
// because rt_load_scene pads every node box by 2^-22 (max |coordinate| + eps),
// which covers the rounding of o * inv; the entry distance is shortened by
// kNearMargin for the relative rounding of both distances.
// ---------------------------------------------------------------------------
// Entry distances are shortened before they are compared with exit and hit
// distances, at the box test and, as the stacks hold them shortened, when an
// entry is popped.  In units of u = 2^-24 of an entry distance, the padding
// leaves uncovered 4 (2 of the four-wide kernels' approximate reciprocal, 1 of
// each rounding after it), and 5 from any origin, whose distance the padding
// does not relate to; the exit distance has the same, and a hit's distance the
// roundings of the triangle test.  Entries popped by the unshortened distance
// dropped boxes that held a hit at an equal or rounding-nearer distance.
constexpr float kNearMargin = 1.0f - 0x1p-21f;     // 8 u
constexpr float kNearMarginAny = 1.0f - 0x1p-20f;  // 16 u: four-wide nodes, any origin
struct Trav {
  RayW rw;
  float3 inv, oinv;
  float best_t;
  uint32_t best_id;
  int best_leaf;
  uint32_t ref, cnt;
  int sp;
  uint32_t iter;
  uint32_t oct;  // four-wide nodes: bit a set when the ray runs towards -axis a
};

template <bool FMA>
__device__ __forceinline__ float box_t(const Trav& tv, float4 lo, float4 hi, float tmax) {
  float tx0, tx1, ty0, ty1, tz0, tz1;
  if (FMA) {
    tx0 = fmaf(lo.x, tv.inv.x, -tv.oinv.x);
    tx1 = fmaf(hi.x, tv.inv.x, -tv.oinv.x);
    ty0 = fmaf(lo.y, tv.inv.y, -tv.oinv.y);
    ty1 = fmaf(hi.y, tv.inv.y, -tv.oinv.y);
    tz0 = fmaf(lo.z, tv.inv.z, -tv.oinv.z);
    tz1 = fmaf(hi.z, tv.inv.z, -tv.oinv.z);
  } else {
    // oinv holds the origin itself in this mode
    tx0 = __fmul_rn(__fsub_rn(lo.x, tv.oinv.x), tv.inv.x);
    tx1 = __fmul_rn(__fsub_rn(hi.x, tv.oinv.x), tv.inv.x);
    ty0 = __fmul_rn(__fsub_rn(lo.y, tv.oinv.y), tv.inv.y);
    ty1 = __fmul_rn(__fsub_rn(hi.y, tv.oinv.y), tv.inv.y);
    tz0 = __fmul_rn(__fsub_rn(lo.z, tv.oinv.z), tv.inv.z);
    tz1 = __fmul_rn(__fsub_rn(hi.z, tv.oinv.z), tv.inv.z);
  }
  const float tn = kNearMargin * fmaxf(fmaxf(fminf(tx0, tx1), fminf(ty0, ty1)), fmaxf(fminf(tz0, tz1), 0.0f));
  const float tf = fminf(fminf(fmaxf(tx0, tx1), fmaxf(ty0, ty1)), fminf(fmaxf(tz0, tz1), tmax));
  return tn <= tf ? tn : -1.0f;
}

// Starts a ray; returns false if it misses the root box (finished).
template <bool FMA>
__device__ __forceinline__ bool trav_init(Trav& tv, const DevScene& S, float3 o, float3 d) {
  tv.rw = ray_prep(o, d);
  const float tiny = 1e-20f;
  tv.inv.x = 1.0f / (fabsf(d.x) > tiny ? d.x : copysignf(tiny, d.x));
  tv.inv.y = 1.0f / (fabsf(d.y) > tiny ? d.y : copysignf(tiny, d.y));
  tv.inv.z = 1.0f / (fabsf(d.z) > tiny ? d.z : copysignf(tiny, d.z));
  tv.oinv = FMA ? make_float3(o.x * tv.inv.x, o.y * tv.inv.y, o.z * tv.inv.z) : o;
  tv.best_t = INFINITY;
  tv.best_id = 0xFFFFFFFFu;
  tv.best_leaf = -1;
  tv.sp = 0;
  tv.iter = 0;
  const float4 rlo = ldg4(S.nodes + 2), rhi = ldg4(S.nodes + 3);
  tv.ref = __float_as_uint(rlo.w);
  tv.cnt = __float_as_uint(rhi.w);
  return box_t<FMA>(tv, rlo, rhi, INFINITY) >= 0.0f;
}

// Interior node: test both children of pair ref, descend into the nearer,
// push the farther.  Returns false if neither child is entered.
template <bool FMA, bool COUNT>
__device__ __forceinline__ bool trav_interior(Trav& tv, uint2* stack, const DevScene& S, float tmax, uint32_t* status,
                                              uint32_t& n_nodes) {
  const float4* c = S.nodes + 2u * tv.ref;
  const float4 alo = ldg4(c), ahi = ldg4(c + 1), blo = ldg4(c + 2), bhi = ldg4(c + 3);
  if (COUNT) n_nodes += 2;
  const float ta = box_t<FMA>(tv, alo, ahi, tmax);
  const float tb = box_t<FMA>(tv, blo, bhi, tmax);
  // branch-free: descend into the nearer entered child; the farther one is
  // written to the stack unconditionally and kept only when both are entered
  const bool ha = ta >= 0.0f, hb = tb >= 0.0f;
  const bool an = ha && (!hb || ta <= tb);
  const bool both = ha && hb;
  if (both && tv.sp >= kStack) {
    atomicOr(status, ST_STACK);
    tv.sp = 0;
    return false;
  }
  const uint32_t fref = __float_as_uint(an ? blo.w : alo.w), fcnt = __float_as_uint(an ? bhi.w : ahi.w);
  stack[min(tv.sp, kStack - 1)] = make_uint2((fref << 3) | fcnt, __float_as_uint(an ? tb : ta));
  tv.sp += both ? 1 : 0;
  tv.ref = __float_as_uint(an ? alo.w : blo.w);
  tv.cnt = __float_as_uint(an ? ahi.w : bhi.w);
  return ha || hb;
}

// Pops the next stack entry whose entry distance is within tmax; false when
// the stack is empty (traversal finished).
__device__ __forceinline__ bool trav_pop(Trav& tv, const uint2* stack, float tmax) {
  while (tv.sp > 0) {
    const uint2 e = stack[--tv.sp];
    if (__uint_as_float(e.y) <= tmax) {
      tv.ref = e.x >> 3;
      tv.cnt = e.x & 7u;
      return true;
    }
  }
  return false;
}

// ---------------------------------------------------------------------------
// Four-wide BVH.  A visit loads the node's three 32-byte sectors (pack_node4).
// With every lane of a warp at another node, these loads bound the kernel as
// much as its instructions do (with four sectors per visit the L1's data path
// was busy in 85% of the cycles, the issue slots in 70%): what counts is how
// many sectors a visit reads and that the lanes' sectors lie in different
// banks.  At a node stride of 128 bytes all lanes read the same quarter of
// their lines and are served one at a time (18 lanes at random nodes in L1: 82
// cycles per visit of four loads, 44 with the quarters permuted from node to
// node); the stride of 96 bytes spreads them by itself.  Closest hits of two
// samples of the 1024 x 768 nave / one of two 1024 x 768 views of the 2M-triangle
// nave: planes in 128 bytes 171.8 / 106.2 ms, quarters permuted and this loop
// 138.2 / 87.4, 96 bytes 128.1 / 81.5, loop parameters swept again 125 / 78;
// sun rays 50.2 / 38.2 -> 36.7 / 29.2.  64-byte nodes on a 15-bit grid gave
// 136.8 / 89.4 against 140.6 / 89.3 of the 128-byte nodes they were tried
// against: a decode per plane costs what the sectors save.
//
// A slab of centre c and half extent h is crossed from (c - o) / d - h / |d| to
// (c - o) / d + h / |d|: no entry and exit plane to select by the ray's sign.
// ---------------------------------------------------------------------------
constexpr uint32_t kIdle = 0xFFFFFFFFu;  // Ray4::cur of a lane without work (no leaf: its count would be 7)

struct Ray4 {
  float3 inv, ainv, oinv;  // 1 / d, |1 / d|, and o / d (FMA box test) or o (any origin)
  float best_t;
  int best_leaf;
  uint32_t cur;  // packed child to visit: ref << 3 | count (count 0: interior node), or kIdle
  uint32_t iter;
};

// What a ray needs only at its leaves or its end lies in shared memory, one
// word per thread and row: the registers it would hold cost resident blocks,
// and each block more per SM is worth 4-5% of the traversal's time.  Row i of
// thread t at word i blockDim.x + t behind `base`.
struct RayRows {
  uint32_t a;  // shared address of the thread's word in row 0
  __device__ __forceinline__ explicit RayRows(uint32_t byte_offset) {
    extern __shared__ __align__(16) unsigned char trav_smem[];
    a = (uint32_t)__cvta_generic_to_shared(trav_smem) + byte_offset + 4u * threadIdx.x;
  }
  __device__ __forceinline__ void put(uint32_t row, uint32_t v) const {
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(a + 4u * blockDim.x * row), "r"(v) : "memory");
  }
  __device__ __forceinline__ void put(uint32_t row, float v) const { put(row, __float_as_uint(v)); }
  __device__ __forceinline__ uint32_t get(uint32_t row) const {
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a + 4u * blockDim.x * row) : "memory");
    return v;
  }
  __device__ __forceinline__ float getf(uint32_t row) const { return __uint_as_float(get(row)); }
  // rows 0-6: the triangle test's form of the ray
  __device__ __forceinline__ void put(const RayW& w) const {
    put(0, w.ox);
    put(1, w.oy);
    put(2, w.oz);
    put(3, w.Sx);
    put(4, w.Sy);
    put(5, w.Sz);
    put(6, (uint32_t)(w.kx | (w.ky << 2) | (w.kz << 4)));
  }
  __device__ __forceinline__ RayW ray() const {
    const uint32_t k = get(6);
    return RayW{getf(0), getf(1), getf(2), (int)(k & 3u), (int)((k >> 2) & 3u), (int)(k >> 4), getf(3), getf(4), getf(5)};
  }
};
constexpr uint32_t kRayRows = 7;
// rows of a sun ray behind those: direction, contribution, path id and flags
constexpr uint32_t kRowDir = 7, kRowContrib = 10, kRowBits = 11, kSunRows = 12;

// FTZ: for unit directions (the paths' own).  A caller's direction past 2^126
// has a reciprocal below the normal range, and 0 in its place would let the
// ray enter every box, the empty ones too.
template <bool FTZ>
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  if (FTZ) asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  else asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float max3f(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float min3f(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// The reciprocals only bound boxes: their 1 ulp error scales both distances
// of a slab alike and is covered by kNearMargin.
template <bool FMA>
__device__ __forceinline__ void ray4_init(Ray4& r, const RayRows& rows, float3 o, float3 d) {
  rows.put(ray_prep(o, d));
  const float tiny = 1e-20f;
  r.inv.x = rcp_approx<FMA>(fabsf(d.x) > tiny ? d.x : copysignf(tiny, d.x));
  r.inv.y = rcp_approx<FMA>(fabsf(d.y) > tiny ? d.y : copysignf(tiny, d.y));
  r.inv.z = rcp_approx<FMA>(fabsf(d.z) > tiny ? d.z : copysignf(tiny, d.z));
  r.oinv = FMA ? make_float3(o.x * r.inv.x, o.y * r.inv.y, o.z * r.inv.z) : o;
  r.ainv = make_float3(fabsf(r.inv.x), fabsf(r.inv.y), fabsf(r.inv.z));
  r.best_t = INFINITY;
  r.best_leaf = -1;
  r.cur = 0u;
  r.iter = 0;
}

// Distances at which the ray enters and leaves the slab of centre c and half
// extent h.  FMA: the rounding of (c - o) / d moves a plane by at most
// 2^-24 (|o| + |c - o|), within the 2^-22 (max |coordinate| + eps) by which
// every box is padded, for origins inside the scene bounds.  Otherwise (any
// origin) the difference first: 4 operations, as many; from the two planes, 8
// with the selects by the ray's sign, a photon pass of the nave took 1.51 ms
// (disk) and 8.70 (portals), this way 1.38 and 7.77; a million closest hits
// 0.297 and 0.262.
template <bool FMA>
__device__ __forceinline__ void slab4(float c, float h, float inv, float ainv, float oinv, float& tn, float& tf) {
  if (FMA) {
    const float tc = fmaf(c, inv, -oinv);
    tn = fmaf(-h, ainv, tc);
    tf = fmaf(h, ainv, tc);
  } else {
    const float tc = __fmul_rn(__fsub_rn(c, oinv), inv);
    tn = fmaf(-h, ainv, tc);
    tf = fmaf(h, ainv, tc);
  }
}

// Half extents of children 0-3 of one axis from their two words.
__device__ __forceinline__ float4 halves(float w01, float w23) {
  return make_float4(__uint_as_float(__float_as_uint(w01) << 16), w01, __uint_as_float(__float_as_uint(w23) << 16), w23);
}

// Entry distance of a child box, +inf if it is missed or begins past tmax.
template <bool FMA>
__device__ __forceinline__ float child4(const Ray4& r, float cx, float hx, float cy, float hy, float cz, float hz,
                                        float tmax) {
  float nx, fx, ny, fy, nz, fz;
  slab4<FMA>(cx, hx, r.inv.x, r.ainv.x, r.oinv.x, nx, fx);
  slab4<FMA>(cy, hy, r.inv.y, r.ainv.y, r.oinv.y, ny, fy);
  slab4<FMA>(cz, hz, r.inv.z, r.ainv.z, r.oinv.z, nz, fz);
  const float tn = (FMA ? kNearMargin : kNearMarginAny) * max3f(nx, ny, fmaxf(nz, 0.0f));
  const float tf = min3f(fx, fy, fminf(fz, tmax));
  return tn <= tf ? tn : INFINITY;
}

__device__ __forceinline__ void cswap(float& ta, uint32_t& pa, float& tb, uint32_t& pb) {
  const bool sw = tb < ta;
  const float t = sw ? tb : ta;
  const uint32_t p = sw ? pb : pa;
  tb = sw ? ta : tb;
  pb = sw ? pa : pb;
  ta = t;
  pa = p;
}

// Traversal stack of one lane for closest hits: the upper entries in shared
// memory (entry j of thread t at column t of row j, so that the lanes of a
// warp never conflict), the rest, which one ray in a thousand reaches, in a
// local array.  From local memory alone 16% of the pops came from L2, on the
// chain between two node visits (nave frame, closest hits: 144.5 ms against
// 140.6 with the shared rows).  An entry is a child and its entry distance.
constexpr uint32_t kRows4 = 6;  // shared entries before the bottom ones move to local memory
constexpr uint32_t kMove4 = 4;  // entries moved at a time
// Shared memory of a block: the stacks (a node pushes at most three entries
// past the rows), then the ray rows.
constexpr uint32_t stack4_bytes(uint32_t block) { return (kRows4 + 3u) * 8u * block; }
constexpr uint32_t trace4_smem(uint32_t block) { return stack4_bytes(block) + kRayRows * 4u * block; }
constexpr uint32_t shadow4_smem(uint32_t block) { return kSunRows * 4u * block; }

struct SharedStack {
  uint32_t top;   // shared address of the first free entry
  uint32_t deep;  // entries in local memory
  uint2* local;   // [kStack + kMove4]
  __device__ __forceinline__ static uint32_t base() {
    extern __shared__ __align__(16) unsigned char trav_smem[];
    return (uint32_t)__cvta_generic_to_shared(trav_smem) + 8u * threadIdx.x;
  }
  __device__ __forceinline__ static uint32_t row() { return 8u * blockDim.x; }
  __device__ __forceinline__ void clear() {
    top = base();
    deep = 0u;
  }
  __device__ __forceinline__ static void put(uint32_t a, uint2 e) {
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(e.x), "r"(e.y) : "memory");
  }
  __device__ __forceinline__ static uint2 get(uint32_t a) {
    uint2 e;
    asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(e.x), "=r"(e.y) : "r"(a) : "memory");
    return e;
  }
  __device__ __forceinline__ void push(uint32_t p, float t) {
    put(top, make_uint2(p, __float_as_uint(t)));
    top += row();
  }
  // After a node's pushes: moves the bottom entries to local memory when the
  // rows are full; false beyond kStack entries.
  __device__ __forceinline__ bool settle() {
    if (top <= base() + kRows4 * row()) return true;
    if (deep + (top - base()) / row() > (uint32_t)kStack) return false;
    uint32_t a = base();
    for (uint32_t j = 0; j < kMove4; ++j, a += row()) local[deep++] = get(a);
    for (; a < top; a += row()) put(a - kMove4 * row(), get(a));
    top -= kMove4 * row();
    return true;
  }
  // The next entry that begins within tmax, or kIdle when none is left.
  __device__ __forceinline__ uint32_t pop(float tmax) {
    for (;;) {
      if (top == base()) {
        if (deep == 0u) return kIdle;
        deep -= kMove4;
        for (uint32_t j = 0; j < kMove4; ++j, top += row()) put(top, local[deep + j]);
      }
      top -= row();
      const uint2 e = get(top);
      if (__uint_as_float(e.y) <= tmax) return e.x;
    }
  }
};

// The same for sun rays, whose entries are children alone: a local array.  A
// sun ray pushes an eighth of what a closest hit does, and the rows cost L1
// (nave frame, sun rays: 38.1 ms, 40.0 with shared rows).
struct LocalStack {
  int sp;
  uint32_t* local;  // [kStack + 3]
  __device__ __forceinline__ void clear() { sp = 0; }
  __device__ __forceinline__ void push(uint32_t p, float) { local[sp++] = p; }
  __device__ __forceinline__ bool settle() const { return sp <= kStack; }
  __device__ __forceinline__ uint32_t pop(float) { return sp > 0 ? local[--sp] : kIdle; }
};

// Interior node r.cur: enters the nearest child that the ray meets and pushes
// the others; false if it meets none.  Three compare-exchanges find the
// nearest child and leave the others nearly sorted (59% of the visits of the
// nave enter one child, 5% more than two: the full order saves 0.4% of the
// visits and costs two exchanges more in each).  ANY (sun rays, which need
// every crossed sheet or one opaque hit, in any order): the entered children
// in slot order, set by k_sun_order4 (farthest along the sun first).
template <bool FMA, bool COUNT, bool ANY, class ST>
__device__ __forceinline__ bool interior4(Ray4& r, ST& stack, const DevScene& S, float tmax, uint32_t* status,
                                          uint32_t& n_nodes) {
  // cur = ref << 3: node at byte 96 ref = 12 cur
  const char* nd = (const char*)S.nodes4 + 12u * (size_t)r.cur;
  float4 cx, cy, cz, a, b, pf;
  ldg8(nd, cx, a);
  ldg8(nd + 32, cy, b);
  ldg8(nd + 64, cz, pf);
  const float4 hx = halves(a.x, a.y), hy = halves(a.z, a.w), hz = halves(b.x, b.y);
  if (COUNT) n_nodes += 4;
  float t0 = child4<FMA>(r, cx.x, hx.x, cy.x, hy.x, cz.x, hz.x, tmax);
  float t1 = child4<FMA>(r, cx.y, hx.y, cy.y, hy.y, cz.y, hz.y, tmax);
  float t2 = child4<FMA>(r, cx.z, hx.z, cy.z, hy.z, cz.z, hz.z, tmax);
  float t3 = child4<FMA>(r, cx.w, hx.w, cy.w, hy.w, cz.w, hz.w, tmax);
  uint32_t p0 = __float_as_uint(pf.x), p1 = __float_as_uint(pf.y), p2 = __float_as_uint(pf.z),
           p3 = __float_as_uint(pf.w);
  if (ANY) {
    // the entered child of the lowest slot stays in cur, the one before goes up
    uint32_t cur = kIdle;
    if (t3 < INFINITY) cur = p3;
    if (t2 < INFINITY) {
      if (cur != kIdle) stack.push(cur, 0.0f);
      cur = p2;
    }
    if (t1 < INFINITY) {
      if (cur != kIdle) stack.push(cur, 0.0f);
      cur = p1;
    }
    if (t0 < INFINITY) {
      if (cur != kIdle) stack.push(cur, 0.0f);
      cur = p0;
    }
    r.cur = cur;
  } else {
    cswap(t0, p0, t1, p1);
    cswap(t2, p2, t3, p3);
    cswap(t0, p0, t2, p2);
    if (t3 < INFINITY) stack.push(p3, t3);
    if (t1 < INFINITY) stack.push(p1, t1);
    if (t2 < INFINITY) stack.push(p2, t2);
    r.cur = t0 < INFINITY ? p0 : kIdle;
  }
  if (!stack.settle()) {
    atomicOr(status, ST_STACK);
    r.cur = kIdle;
    stack.clear();
  }
  return r.cur != kIdle;
}

// The wide variants below (8-bit boxes, eight children) test lo and hi planes,
// the entry and exit plane picked by the ray's direction signs.
template <bool FMA>
__device__ __forceinline__ float slab(float plane, float inv, float oinv) {
  // robust mode: oinv holds the origin itself
  return FMA ? fmaf(plane, inv, -oinv) : __fmul_rn(__fsub_rn(plane, oinv), inv);
}

template <bool FMA>
__device__ __forceinline__ float child_t(const Trav& tv, float nx, float fx, float ny, float fy, float nz, float fz,
                                         float tmax) {
  const float tn = kNearMargin * fmaxf(fmaxf(slab<FMA>(nx, tv.inv.x, tv.oinv.x), slab<FMA>(ny, tv.inv.y, tv.oinv.y)),
                                       fmaxf(slab<FMA>(nz, tv.inv.z, tv.oinv.z), 0.0f));
  const float tf = fminf(fminf(slab<FMA>(fx, tv.inv.x, tv.oinv.x), slab<FMA>(fy, tv.inv.y, tv.oinv.y)),
                         fminf(slab<FMA>(fz, tv.inv.z, tv.oinv.z), tmax));
  return tn <= tf ? tn : INFINITY;
}

template <bool FMA>
__device__ __forceinline__ void trav_init_wide(Trav& tv, float3 o, float3 d) {
  tv.rw = ray_prep(o, d);
  const float tiny = 1e-20f;
  tv.inv.x = 1.0f / (fabsf(d.x) > tiny ? d.x : copysignf(tiny, d.x));
  tv.inv.y = 1.0f / (fabsf(d.y) > tiny ? d.y : copysignf(tiny, d.y));
  tv.inv.z = 1.0f / (fabsf(d.z) > tiny ? d.z : copysignf(tiny, d.z));
  tv.oinv = FMA ? make_float3(o.x * tv.inv.x, o.y * tv.inv.y, o.z * tv.inv.z) : o;
  tv.best_t = INFINITY;
  tv.best_id = 0xFFFFFFFFu;
  tv.best_leaf = -1;
  tv.sp = 0;
  tv.iter = 0;
  tv.ref = 0;
  tv.cnt = 0;
  tv.oct = (tv.inv.x < 0.0f ? 1u : 0u) | (tv.inv.y < 0.0f ? 2u : 0u) | (tv.inv.z < 0.0f ? 4u : 0u);
}

// ---------------------------------------------------------------------------
// Four-wide BVH with 8-bit child boxes (node = 4 float4, 64 bytes: {origin,
// bits(e_x | e_y << 8 | e_z << 16)}, {lo x, hi x, lo y, hi y} and {lo z,
// hi z} as one byte per child, then the children packed as in the float
// node).  Plane q of axis a lies at origin_a + q 2^e_a; the byte becomes the
// float 2^23 + q by a byte permute, and t = fma(2^23 + q, 2^e inv,
// b - 2^23 2^e inv) with b = (origin - o) inv: the subtraction rounds by
// at most half a cell, inside the cell of margin the builder leaves around
// every child box.  Same children, same order, half the bytes per node
// visit of the float node (the closest-hit kernel is bound by L1
// throughput).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float qplane(uint32_t word, uint32_t sel) {
  return __uint_as_float(__byte_perm(word, 0x4B000000u, sel));
}

template <bool FMA>
__device__ __forceinline__ float qslab_base(float origin, float inv, float oinv) {
  return FMA ? fmaf(origin, inv, -oinv) : __fmul_rn(__fsub_rn(origin, oinv), inv);
}

template <bool FMA, bool COUNT>
__device__ __forceinline__ bool trav_interior4q(Trav& tv, uint2* stack, const DevScene& S, float tmax,
                                                uint32_t* status, uint32_t& n_nodes) {
  const float4* nd = S.nodes4q + 4u * tv.ref;
  const float4 h = ldg4(nd), pa = ldg4(nd + 1), pb = ldg4(nd + 2);
  const uint4 pk = __ldg((const uint4*)(nd + 3));
  if (COUNT) n_nodes += 4;
  const uint32_t eb = __float_as_uint(h.w);
  // per axis: cell size times 1/d, and the offset of plane 2^23 + q
  const float sx = __uint_as_float(((eb & 0xFFu) + 127u - ((eb & 0x80u) << 1)) << 23) * tv.inv.x;
  const float sy = __uint_as_float((((eb >> 8) & 0xFFu) + 127u - (((eb >> 8) & 0x80u) << 1)) << 23) * tv.inv.y;
  const float sz = __uint_as_float((((eb >> 16) & 0xFFu) + 127u - (((eb >> 16) & 0x80u) << 1)) << 23) * tv.inv.z;
  const float bx = fmaf(-8388608.0f, sx, qslab_base<FMA>(h.x, tv.inv.x, tv.oinv.x));
  const float by = fmaf(-8388608.0f, sy, qslab_base<FMA>(h.y, tv.inv.y, tv.oinv.y));
  const float bz = fmaf(-8388608.0f, sz, qslab_base<FMA>(h.z, tv.inv.z, tv.oinv.z));
  // near planes: lo when the ray runs towards +axis
  const uint32_t wlx = __float_as_uint(pa.x), whx = __float_as_uint(pa.y);
  const uint32_t wly = __float_as_uint(pa.z), why = __float_as_uint(pa.w);
  const uint32_t wlz = __float_as_uint(pb.x), whz = __float_as_uint(pb.y);
  const uint32_t nx = (tv.oct & 1u) ? whx : wlx, fx = (tv.oct & 1u) ? wlx : whx;
  const uint32_t ny = (tv.oct & 2u) ? why : wly, fy = (tv.oct & 2u) ? wly : why;
  const uint32_t nz = (tv.oct & 4u) ? whz : wlz, fz = (tv.oct & 4u) ? wlz : whz;
  float t[4];
#pragma unroll
  for (uint32_t i = 0; i < 4; ++i) {
    const uint32_t sel = 0x7540u | i;
    const float tn = kNearMargin * fmaxf(fmaxf(fmaf(qplane(nx, sel), sx, bx), fmaf(qplane(ny, sel), sy, by)),
                                         fmaxf(fmaf(qplane(nz, sel), sz, bz), 0.0f));
    const float tf = fminf(fminf(fmaf(qplane(fx, sel), sx, bx), fmaf(qplane(fy, sel), sy, by)),
                           fminf(fmaf(qplane(fz, sel), sz, bz), tmax));
    t[i] = tn <= tf ? tn : INFINITY;
  }
  float t0 = t[0], t1 = t[1], t2 = t[2], t3 = t[3];
  uint32_t p0 = pk.x, p1 = pk.y, p2 = pk.z, p3 = pk.w;
  const int nh = (t0 < INFINITY) + (t1 < INFINITY) + (t2 < INFINITY) + (t3 < INFINITY);
  if (nh == 0) return false;
  cswap(t0, p0, t1, p1);
  cswap(t2, p2, t3, p3);
  cswap(t0, p0, t2, p2);
  cswap(t1, p1, t3, p3);
  cswap(t1, p1, t2, p2);
  if (tv.sp + nh - 1 > kStack) {
    atomicOr(status, ST_STACK);
    tv.sp = 0;
    return false;
  }
  const int top = tv.sp + nh - 2;
  if (nh > 1) stack[top] = make_uint2(p1, __float_as_uint(t1));
  if (nh > 2) stack[top - 1] = make_uint2(p2, __float_as_uint(t2));
  if (nh > 3) stack[top - 2] = make_uint2(p3, __float_as_uint(t3));
  tv.sp += nh - 1;
  tv.ref = p0 >> 3;
  tv.cnt = p0 & 7u;
  return true;
}

// ---------------------------------------------------------------------------
// Eight-wide BVH (node = 14 float4: per axis the lo planes of children 0-3
// and 4-7, then their hi planes, then the eight children packed as
// ref << 3 | count).  The builder puts in slot s the child that lies towards
// the corner ((s & 1) ? +x : -x, (s & 2) ? +y : -y, (s & 4) ? +z : -z) of the
// node, so visiting the entered children in the order s = i ^ oct meets the
// corner nearest to the ray first without a per-ray sort: the first entered
// child in that order is descended into, the others pushed with the next one
// on top.  Half a node (children 0-3, then 4-7) is tested at a time.
// ---------------------------------------------------------------------------
template <bool FMA, bool COUNT>
__device__ __forceinline__ bool trav_interior8(Trav& tv, uint2* stack, const DevScene& S, float tmax,
                                               uint32_t* status, uint32_t& n_nodes) {
  const float4* nd = S.nodes8 + 14u * tv.ref;
  const uint32_t ox = (tv.oct & 1u) << 1, oy = tv.oct & 2u, oz = (tv.oct >> 1) & 2u;
  if (COUNT) n_nodes += 8;
  float t[8];
#pragma unroll
  for (uint32_t h = 0; h < 2; ++h) {
    const float4 nx = ldg4(nd + ox + h), fx = ldg4(nd + (ox ^ 2u) + h);
    const float4 ny = ldg4(nd + 4u + oy + h), fy = ldg4(nd + 4u + (oy ^ 2u) + h);
    const float4 nz = ldg4(nd + 8u + oz + h), fz = ldg4(nd + 8u + (oz ^ 2u) + h);
    t[4 * h] = child_t<FMA>(tv, nx.x, fx.x, ny.x, fy.x, nz.x, fz.x, tmax);
    t[4 * h + 1] = child_t<FMA>(tv, nx.y, fx.y, ny.y, fy.y, nz.y, fz.y, tmax);
    t[4 * h + 2] = child_t<FMA>(tv, nx.z, fx.z, ny.z, fy.z, nz.z, fz.z, tmax);
    t[4 * h + 3] = child_t<FMA>(tv, nx.w, fx.w, ny.w, fy.w, nz.w, fz.w, tmax);
  }
  uint32_t m = 0;
#pragma unroll
  for (int s = 0; s < 8; ++s) m |= (t[s] < INFINITY ? 1u : 0u) << s;
  if (m == 0u) return false;
  const int nh = __popc(m);
  if (tv.sp + nh - 1 > kStack) {
    atomicOr(status, ST_STACK);
    tv.sp = 0;
    return false;
  }
  const uint4 pa = __ldg((const uint4*)(nd + 12)), pb = __ldg((const uint4*)(nd + 13));
  const uint32_t p[8] = {pa.x, pa.y, pa.z, pa.w, pb.x, pb.y, pb.z, pb.w};
  // the entered slots in visit order: bit i of v is slot i ^ oct
  uint32_t v = m;
  if (tv.oct & 1u) v = ((v & 0x55u) << 1) | ((v >> 1) & 0x55u);
  if (tv.oct & 2u) v = ((v & 0x33u) << 2) | ((v >> 2) & 0x33u);
  if (tv.oct & 4u) v = ((v & 0x0Fu) << 4) | ((v >> 4) & 0x0Fu);
  // visit rank r >= 1 goes to stack[top - r], rank 1 on top
  const int top = tv.sp + nh - 1;
#pragma unroll
  for (int s = 0; s < 8; ++s) {
    if (t[s] < INFINITY) {
      const uint32_t i = (uint32_t)s ^ tv.oct;
      const int r = __popc(v & ((1u << i) - 1u));
      if (r == 0) {
        tv.ref = p[s] >> 3;
        tv.cnt = p[s] & 7u;
      } else {
        stack[top - r] = make_uint2(p[s], __float_as_uint(t[s]));
      }
    }
  }
  tv.sp += nh - 1;
  return true;
}

// Starts a ray (WIDE: the eight-wide and 8-bit variants); false if it misses
// the binary tree's root box.
template <bool WIDE, bool FMA>
__device__ __forceinline__ bool init_w(Trav& tv, const DevScene& S, float3 o, float3 d) {
  if (WIDE) {
    trav_init_wide<FMA>(tv, o, d);
    return true;
  }
  return trav_init<FMA>(tv, S, o, d);
}

__device__ __forceinline__ void closest_leaf(Trav& tv, const DevScene& S, uint32_t& n_tris, bool count) {
  for (uint32_t t = tv.ref; t < tv.ref + tv.cnt; ++t) {
    const float4* tr = S.tris + 3u * t;
    if (count) ++n_tris;
    const float th = tri_hit(tv.rw, tr);
    const uint32_t id = __float_as_uint(__ldg(&tr->w));
    if (th > 0.0f && (th < tv.best_t || (th == tv.best_t && id < tv.best_id))) {
      tv.best_t = th;
      tv.best_leaf = (int)t;
      tv.best_id = id;
    }
  }
}

__device__ __forceinline__ uint32_t tri_id(const DevScene& S, uint32_t t) {
  return __float_as_uint(__ldg(&S.tris[3 * (size_t)t].w));
}

// The same for Ray4, which reads the ids only on a tie in t.
__device__ __forceinline__ void closest_leaf4(Ray4& r, const RayRows& rows, const DevScene& S, uint32_t& n_tris,
                                              bool count) {
  const RayW w = rows.ray();
  const uint32_t ref = r.cur >> 3, end = ref + (r.cur & 7u);
  for (uint32_t t = ref; t < end; ++t) {
    if (count) ++n_tris;
    const float th = tri_hit(w, S.tris + 3u * t);
    if (th > 0.0f && th <= r.best_t &&
        (th < r.best_t || r.best_leaf < 0 || tri_id(S, t) < tri_id(S, (uint32_t)r.best_leaf))) {
      r.best_t = th;
      r.best_leaf = (int)t;
    }
  }
}

// One closest-hit step (t > 0; ties in t go to the lower input id).  With WW
// (Aila and Laine's while-while form) the step runs interior nodes until the
// lane reaches a leaf, then that leaf, so that a warp's lanes execute the same
// phase together.
template <bool FMA, bool COUNT, bool WW>
__device__ __forceinline__ bool closest_step(Trav& tv, uint2* stack, const DevScene& S, uint32_t cap,
                                             uint32_t* status, uint32_t& n_nodes, uint32_t& n_tris) {
  if (WW) {
    while (tv.cnt == 0u) {
      if (++tv.iter > cap) {
        atomicOr(status, ST_ITER);
        return true;
      }
      if (!trav_interior<FMA, COUNT>(tv, stack, S, tv.best_t, status, n_nodes) && !trav_pop(tv, stack, tv.best_t))
        return true;
    }
    closest_leaf(tv, S, n_tris, COUNT);
    return !trav_pop(tv, stack, tv.best_t);
  }
  if (++tv.iter > cap) {
    atomicOr(status, ST_ITER);
    return true;
  }
  if (tv.cnt == 0u) {
    if (trav_interior<FMA, COUNT>(tv, stack, S, tv.best_t, status, n_nodes)) return false;
  } else {
    closest_leaf(tv, S, n_tris, COUNT);
  }
  return !trav_pop(tv, stack, tv.best_t);
}

// Sun-ray leaf: product of thin-glass T_s over every crossed sheet; returns
// true at the first opaque triangle (T = 0, n_glass = 0xFFFFFFFF).
__device__ __forceinline__ bool shadow_leaf(const RayW& rw, const DevScene& S, const DevSpectra& P, float3 d,
                                            uint32_t ref, uint32_t cnt, uint32_t band, float& T, uint32_t& ng,
                                            uint32_t& n_tris, bool count) {
  for (uint32_t t = ref; t < ref + cnt; ++t) {
    const float4* tr = S.tris + 3u * t;
    if (count) ++n_tris;
    const float th = tri_hit(rw, tr);
    if (th > 0.0f) {
      const uint32_t mat = __float_as_uint(__ldg(&tr[1].w));
      if (__ldg(P.mtype + mat) != 1) {
        T = 0.0f;
        ng = 0xFFFFFFFFu;
        return true;
      }
      const float4 nr = ldg4(S.nrm + t);
      const float c = fabsf(dot(d, f3(nr)));
      const float4 m = ldg4(P.mb + mat * P.n_bands + band);
      float Rs, Ts;
      thin_sheet(c, m.x, m.y, __ldg(P.ad + mat * P.n_bands + band), Rs, Ts);
      T *= Ts;
      ++ng;
    }
  }
  return false;
}

// Sun-ray leaf of the four-wide kernel: as above, for the one band (NB = 1) or
// the four bands band + q G (those the path carries) of the ray's path.  The
// direction and the path are read at a crossed sheet only.
template <int NB>
__device__ __forceinline__ bool shadow_leaf4w(const RayRows& rows, const DevScene& S, const DevSpectra& P,
                                              const WaveParams& w, uint32_t ref, uint32_t cnt, float (&T)[NB],
                                              uint32_t& ng, uint32_t& n_tris, bool count) {
  const RayW rw = rows.ray();
  for (uint32_t t = ref; t < ref + cnt; ++t) {
    const float4* tr = S.tris + 3u * t;
    if (count) ++n_tris;
    const float th = tri_hit(rw, tr);
    if (th > 0.0f) {
      const uint32_t mat = __float_as_uint(__ldg(&tr[1].w));
      if (__ldg(P.mtype + mat) != 1) {
#pragma unroll
        for (int q = 0; q < NB; ++q) T[q] = 0.0f;
        ng = 0xFFFFFFFFu;
        return true;
      }
      const float4 nr = ldg4(S.nrm + t);
      const float3 d = make_float3(rows.getf(kRowDir), rows.getf(kRowDir + 1), rows.getf(kRowDir + 2));
      const float c = fabsf(dot(d, f3(nr)));
      const uint32_t j = path_id(w, rows.get(kRowBits) & kPidMask).j;
      const uint32_t nv = NB == 4 ? four_band_count(w, j) : 1u;
#pragma unroll
      for (uint32_t q = 0; q < (uint32_t)NB; ++q)
        if (q < nv) {
          const uint32_t mb = mat * P.n_bands + w.band_first + j + q * w.band_count;
          const float4 m = ldg4(P.mb + mb);
          float Rs, Ts;
          thin_sheet(c, m.x, m.y, __ldg(P.ad + mb), Rs, Ts);
          T[q] *= Ts;
        }
      ++ng;
    }
  }
  return false;
}

// One sun-ray step (WW as for closest_step).
template <bool FMA, bool COUNT, bool WW>
__device__ __forceinline__ bool shadow_step(Trav& tv, uint2* stack, const DevScene& S, const DevSpectra& P, float3 d,
                                            uint32_t band, float& T, uint32_t& ng, uint32_t cap, uint32_t* status,
                                            uint32_t& n_nodes, uint32_t& n_tris) {
  if (WW) {
    while (tv.cnt == 0u) {
      if (++tv.iter > cap) {
        atomicOr(status, ST_ITER);
        return true;
      }
      if (!trav_interior<FMA, COUNT>(tv, stack, S, INFINITY, status, n_nodes) && !trav_pop(tv, stack, INFINITY))
        return true;
    }
    if (shadow_leaf(tv.rw, S, P, d, tv.ref, tv.cnt, band, T, ng, n_tris, COUNT)) return true;
    return !trav_pop(tv, stack, INFINITY);
  }
  if (++tv.iter > cap) {
    atomicOr(status, ST_ITER);
    return true;
  }
  if (tv.cnt == 0u) {
    if (trav_interior<FMA, COUNT>(tv, stack, S, INFINITY, status, n_nodes)) return false;
  } else {
    if (shadow_leaf(tv.rw, S, P, d, tv.ref, tv.cnt, band, T, ng, n_tris, COUNT)) return true;
  }
  return !trav_pop(tv, stack, INFINITY);
}

__device__ __forceinline__ uint32_t trav_cap(const DevScene& S) {
  return S.iter_cap ? S.iter_cap : 4u * S.n_nodes + 64u;
}

// Whole-ray helpers (any origin).
__device__ __forceinline__ void closest_hit(const DevScene& S, float3 o, float3 d, float& best_t, int& best_leaf,
                                            uint32_t* status) {
  Ray4 r;
  uint2 local[kStack + kMove4];
  SharedStack stack;
  stack.local = local;
  const RayRows rows(stack4_bytes(blockDim.x));
  uint32_t a = 0, b = 0;
  stack.clear();
  ray4_init<false>(r, rows, o, d);
  const uint32_t cap = trav_cap(S);
  while (r.cur != kIdle) {
    if (++r.iter > cap) {
      atomicOr(status, ST_ITER);
      break;
    }
    if ((r.cur & 7u) == 0u) {
      if (interior4<false, false, false>(r, stack, S, r.best_t, status, a)) continue;
    } else {
      closest_leaf4(r, rows, S, b, false);
    }
    r.cur = stack.pop(r.best_t);
  }
  best_t = r.best_t;
  best_leaf = r.best_leaf;
}

__device__ __forceinline__ float shadow_T(const DevScene& S, const DevSpectra& P, float3 o, float3 d, uint32_t band,
                                          uint32_t& n_glass, uint32_t* status) {
  Ray4 r;
  uint32_t local[kStack + 3];
  LocalStack stack;
  stack.local = local;
  uint32_t a = 0, b = 0;
  float T = 1.0f;
  uint32_t ng = 0;
  const RayRows rows(0u);
  stack.clear();
  ray4_init<false>(r, rows, o, d);
  const uint32_t cap = trav_cap(S);
  while (r.cur != kIdle) {
    if (++r.iter > cap) {
      atomicOr(status, ST_ITER);
      break;
    }
    if ((r.cur & 7u) == 0u) {
      if (interior4<false, false, true>(r, stack, S, INFINITY, status, a)) continue;
    } else if (shadow_leaf(rows.ray(), S, P, d, r.cur >> 3, r.cur & 7u, band, T, ng, b, false)) {
      break;
    }
    r.cur = stack.pop(INFINITY);
  }
  n_glass = ng;
  return T;
}

// Exclusive prefix sum of the bins: each block of 1024 threads scans one
// chunk of 1024 bins in place and writes the chunk total; the chunk totals
// (kCellSortBins / 1024 of them) are then scanned by one block, and the
// scatter adds the chunk's offset.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* warp_sums, uint32_t& total) {
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (uint32_t o = 1; o < 32u; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31u) warp_sums[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < nw ? warp_sums[lane] : 0u;
#pragma unroll
    for (uint32_t o = 1; o < 32u; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) warp_sums[lane] = w;  // inclusive over warps
  }
  __syncthreads();
  total = warp_sums[nw - 1];
  const uint32_t before = warp == 0 ? 0u : warp_sums[warp - 1];
  return before + x - v;
}

__global__ void __launch_bounds__(1024) k_cell_scan_chunks(uint32_t* __restrict__ bins, uint32_t* __restrict__ totals) {
  __shared__ uint32_t ws[32];
  const uint32_t i = blockIdx.x * 1024u + threadIdx.x;
  uint32_t tot;
  const uint32_t ex = block_exclusive_scan(bins[i], ws, tot);
  bins[i] = ex;
  if (threadIdx.x == 0) totals[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(1024) k_cell_scan_totals(uint32_t* __restrict__ totals) {
  __shared__ uint32_t ws[32];
  uint32_t tot;
  const uint32_t ex = block_exclusive_scan(totals[threadIdx.x], ws, tot);
  __syncthreads();
  totals[threadIdx.x] = ex;
}

// ---------------------------------------------------------------------------
// Cell sort of a ray queue (counting sort, 2^18 keys): vertex >= 2 rays by
// the Morton cell of their origin on a 32^3 grid over the scene box and
// their direction octant, sun rays (all nearly parallel) by the Morton cell
// on a 64^3 grid.  Rays of one warp then start close together and share the
// nodes they fetch.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t morton3(uint32_t x, uint32_t y, uint32_t z, uint32_t bits) {
  uint32_t r = 0;
  for (uint32_t b = 0; b < bits; ++b)
    r |= (((x >> b) & 1u) << (3u * b)) | (((y >> b) & 1u) << (3u * b + 1u)) | (((z >> b) & 1u) << (3u * b + 2u));
  return r;
}

__device__ __forceinline__ uint32_t cell_of(const DevScene& S, float3 o, uint32_t bits) {
  const float n = (float)(1u << bits);
  const uint32_t m = (1u << bits) - 1u;
  const uint32_t x = min((uint32_t)fmaxf((o.x - S.blo[0]) * S.binv[0] * n, 0.0f), m);
  const uint32_t y = min((uint32_t)fmaxf((o.y - S.blo[1]) * S.binv[1] * n, 0.0f), m);
  const uint32_t z = min((uint32_t)fmaxf((o.z - S.blo[2]) * S.binv[2] * n, 0.0f), m);
  return morton3(x, y, z, bits);
}

template <bool SUN>
__global__ void k_rsort_hist(DevScene S, const float4* __restrict__ q, const Counters* __restrict__ cnt, uint32_t k,
                             uint32_t cap, uint32_t* __restrict__ key, uint32_t* __restrict__ bins) {
  const uint32_t count = min(SUN ? cnt[k].s_count : cnt[k].q_count, cap);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const float4 a = __ldg(q + 2 * i);
    uint32_t kk;
    if (SUN) {
      kk = cell_of(S, f3(a), 6u);
    } else {
      const float4 b = __ldg(q + 2 * i + 1);
      const uint32_t oct = (b.x < 0.0f ? 1u : 0u) | (b.y < 0.0f ? 2u : 0u) | (b.z < 0.0f ? 4u : 0u);
      kk = cell_of(S, f3(a), 5u) | (oct << 15);
    }
    key[i] = kk;
    atomicAdd(bins + kk, 1u);
  }
}

template <bool SUN>
__global__ void k_rsort_scatter(const Counters* __restrict__ cnt, uint32_t k, uint32_t cap,
                                const uint32_t* __restrict__ key, uint32_t* __restrict__ bins,
                                uint32_t* __restrict__ perm) {
  const uint32_t count = min(SUN ? cnt[k].s_count : cnt[k].q_count, cap);
  const uint32_t* totals = bins + kCellSortBins;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
    const uint32_t kk = key[i];
    perm[__ldg(totals + (kk >> 10)) + atomicAdd(bins + kk, 1u)] = i;
  }
}

// ---------------------------------------------------------------------------
// kernels
// ---------------------------------------------------------------------------

__global__ void __launch_bounds__(256) k_camera(const DevCam* __restrict__ cams, uint32_t n_cams, WaveParams w,
                                                float4* __restrict__ q, float* __restrict__ L,
                                                uint32_t* __restrict__ sig, Counters* cnt, bool record,
                                                float4* __restrict__ L4, float4* __restrict__ T4, uint32_t cap,
                                                uint32_t* status) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    cnt[1].q_count = w.n;
    if (w.n > cap) atomicOr(status, ST_QUEUE);  // a wave larger than its ray queue
  }
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < w.n; i += stride) {
    const PathId id = path_id(w, i);
    uint32_t v = 0;
    while (v + 1 < n_cams && cams[v + 1].offset <= id.pix) ++v;
    const DevCam& C = cams[v];
    const uint32_t local = id.pix - C.offset;
    const uint32_t y = local / C.W, x = local - y * C.W;
    const uint4 u = philox4x32_10(make_uint4(id.pix, id.s, w.band_first + id.j, 0u), w.key0, w.key1);
    const float sx = (2.0f * ((float)x + u01(u.x)) / (float)C.W - 1.0f) * C.tha;
    const float sy = (1.0f - 2.0f * ((float)y + u01(u.y)) / (float)C.H) * C.th;
    float3 dir = make_float3(C.f.x + sx * C.r.x + sy * C.u.x, C.f.y + sx * C.r.y + sy * C.u.y,
                             C.f.z + sx * C.r.z + sy * C.u.z);
    const float inv = 1.0f / sqrtf(dot(dir, dir));
    dir = mul(inv, dir);
    q[2 * i] = make_float4(C.pos.x, C.pos.y, C.pos.z, __uint_as_float(i));
    q[2 * i + 1] = make_float4(dir.x, dir.y, dir.z, 1.0f);
    if (w.nb == 4u) {
      // bands past the render's range carry nothing
      const uint32_t nv = four_band_count(w, id.j);
      L4[i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      T4[i] = make_float4(1.0f, nv > 1u ? 1.0f : 0.0f, nv > 2u ? 1.0f : 0.0f, nv > 3u ? 1.0f : 0.0f);
    } else {
      L[i] = 0.0f;
    }
    if (record) sig[i] = 2166136261u;
  }
}

constexpr uint32_t kNoRay = 0xFFFFFFFFu;
// The kernels over the other trees (trace_variant 1 to 5): blocks of at most
// 128 threads, launch bound 8 blocks per SM (<= 64 registers, none spilled).
#ifndef SRT_TRACE_MIN_BLOCKS
#define SRT_TRACE_MIN_BLOCKS 8
#endif
constexpr int kTraceMaxThreads = 128, kTraceMinBlocks = SRT_TRACE_MIN_BLOCKS;
// four-wide kernels: 9 blocks of 128 per SM (<= 56 registers, none spilled).
// Two samples of the 1024 x 768 nave / one of two 1024 x 768 views of the
// 2M-triangle nave, closest hits: 9 blocks 128.1 / 81.5 ms, 10 (48 registers)
// 130.0 / 82.3; sun rays 36.7 / 29.2, 8 blocks 37.8 / 30.1, 10 36.4 / 29.2.
constexpr int kTrace4MinBlocks = 9, kShadow4MinBlocks = 9;
// Persistent traversal loop: a warp refills its idle lanes from the queue
// once at least `refill` lanes are idle, and each lane with a ray runs up to
// `steps` traversal steps between refill checks (steps large and refill 32
// give one batch of 32 rays per warp at a time).

// MODE 0: each lane runs up to `steps` node-or-leaf steps; 1: while-while
// steps; 2: warp-synchronous phases - interior steps for the lanes at an
// interior node until at least `leaf_min` lanes wait at a leaf (or none can
// go on), then one leaf step for every waiting lane, so that the costly
// triangle tests run with most of their lanes busy; 4 and 5 (trace_variant 4,
// 5): as 2 over the eight-wide BVH and the 8-bit four-wide one.  Modes 0-2
// traverse the binary BVH; k_trace4 below, the default, the four-wide one.
template <bool FMA, bool COUNT, int MODE>
__global__ void __launch_bounds__(kTraceMaxThreads, kTraceMinBlocks) k_trace(DevScene S, const float4* __restrict__ q, float2* __restrict__ hit,
                                               Counters* cnt, uint32_t k, uint32_t cap, Totals* tot,
                                               uint32_t* status, int steps, int refill, int leaf_min,
                                               const uint32_t* __restrict__ perm) {
  const uint32_t count = min(cnt[k].q_count, cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&tot->ext_rays, (unsigned long long)count);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t icap = trav_cap(S);
  uint32_t nn = 0, nt = 0;
  Trav tv;
  uint2 stack[kStack];
  uint32_t ray = kNoRay;
  bool drained = count == 0u;
  for (;;) {
    const uint32_t idle = __ballot_sync(0xffffffffu, ray == kNoRay);
    if (!drained && (int)__popc(idle) >= refill) {
      const uint32_t n = __popc(idle);
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(&cnt[k].q_fetch, n);
      base = __shfl_sync(0xffffffffu, base, 0);
      if (base + n >= count) drained = true;
      if (ray == kNoRay) {
        const uint32_t slot = base + __popc(idle & lt);
        if (slot < count) {
          const uint32_t ri = perm ? __ldg(perm + slot) : slot;
          const float4 a = __ldcs(q + 2 * ri), b = __ldcs(q + 2 * ri + 1);
          if (init_w<MODE >= 4, FMA>(tv, S, f3(a), f3(b))) {
            ray = ri;
          } else {
            __stcs(hit + ri, make_float2(-1.0f, __int_as_float(-1)));
          }
        }
      }
    }
    if (!__any_sync(0xffffffffu, ray != kNoRay)) {
      if (drained) break;
      continue;
    }
    if (MODE >= 2) {
      bool done = false;
      for (int i = 0; i < steps; ++i) {
        const bool act = ray != kNoRay && !done;
        const bool at_leaf = act && tv.cnt != 0u;
        const uint32_t ml = __ballot_sync(0xffffffffu, at_leaf);
        const uint32_t mi = __ballot_sync(0xffffffffu, act && !at_leaf);
        if ((ml | mi) == 0u) break;
        const bool leaf_phase = mi == 0u || (int)__popc(ml) >= leaf_min;
        if (act && at_leaf == leaf_phase) {
          if (++tv.iter > icap) {
            atomicOr(status, ST_ITER);
            done = true;
          } else if (leaf_phase) {
            closest_leaf(tv, S, nt, COUNT);
            done = !trav_pop(tv, stack, tv.best_t);
          } else if (!(MODE == 5   ? trav_interior4q<FMA, COUNT>(tv, stack, S, tv.best_t, status, nn)
                       : MODE == 4 ? trav_interior8<FMA, COUNT>(tv, stack, S, tv.best_t, status, nn)
                                   : trav_interior<FMA, COUNT>(tv, stack, S, tv.best_t, status, nn))) {
            done = !trav_pop(tv, stack, tv.best_t);
          }
        }
      }
      if (ray != kNoRay && done) {
        __stcs(hit + ray, make_float2(tv.best_leaf < 0 ? -1.0f : tv.best_t, __int_as_float(tv.best_leaf)));
        ray = kNoRay;
      }
    } else if (ray != kNoRay) {
      bool done = false;
      for (int i = 0; i < steps && !done; ++i)
        done = closest_step<FMA, COUNT, MODE == 1>(tv, stack, S, icap, status, nn, nt);
      if (done) {
        __stcs(hit + ray, make_float2(tv.best_leaf < 0 ? -1.0f : tv.best_t, __int_as_float(tv.best_leaf)));
        ray = kNoRay;
      }
    }
  }
  if (COUNT) {
    atomicAdd(&tot->nodes, (unsigned long long)nn);
    atomicAdd(&tot->tris, (unsigned long long)nt);
  }
}

// Closest hits over the four-wide BVH (render option trace_variant 0):
// persistent warps refill idle lanes from the queue; a warp runs interior
// steps for its lanes at interior nodes until at least leaf_min lanes wait at
// a leaf (or none can go on), then one leaf step for every waiting lane.  The
// loop's own instructions weigh as much as a box test, so each step takes one
// vote, and the step limit is checked between rounds of `steps`.
template <bool FMA, bool COUNT>
__global__ void __launch_bounds__(kTraceMaxThreads, kTrace4MinBlocks)
    k_trace4(DevScene S, const float4* __restrict__ q, float2* __restrict__ hit, Counters* cnt, uint32_t k, uint32_t cap,
             Totals* tot, uint32_t* status, int steps, int refill, int leaf_min, const uint32_t* __restrict__ perm) {
  const uint32_t count = min(cnt[k].q_count, cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&tot->ext_rays, (unsigned long long)count);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t icap = trav_cap(S);
  uint32_t nn = 0, nt = 0;
  Ray4 r;
  uint2 local[kStack + kMove4];
  SharedStack stack;
  stack.local = local;
  stack.clear();
  const RayRows rows(stack4_bytes(blockDim.x));
  uint32_t ray = kNoRay;
  r.cur = kIdle;
  bool drained = count == 0u;
  for (;;) {
    const uint32_t idle = __ballot_sync(0xffffffffu, ray == kNoRay);
    if (!drained && (int)__popc(idle) >= refill) {
      const uint32_t n = __popc(idle);
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(&cnt[k].q_fetch, n);
      base = __shfl_sync(0xffffffffu, base, 0);
      if (base + n >= count) drained = true;
      const uint32_t slot = base + __popc(idle & lt);
      if (ray == kNoRay && slot < count) {
        ray = perm ? __ldg(perm + slot) : slot;
        const float4 a = __ldcs(q + 2 * ray), b = __ldcs(q + 2 * ray + 1);
        ray4_init<FMA>(r, rows, f3(a), f3(b));
      }
    } else if (idle == 0xffffffffu) {
      break;  // drained
    }
    // a leaf step once all but this many of the lanes with a ray have left
    // the interior (they wait at a leaf, or have finished in this round)
    const int nodes_min = (int)__popc(__ballot_sync(0xffffffffu, ray != kNoRay)) - leaf_min;
    for (int i = 0; i < steps; ++i) {
      const bool at_node = (r.cur & 7u) == 0u;
      const bool at_leaf = !at_node && r.cur != kIdle;
      const uint32_t mi = __ballot_sync(0xffffffffu, at_node);
      if (mi == 0u || (int)__popc(mi) <= nodes_min) {
        if (!__any_sync(0xffffffffu, at_leaf)) break;  // none left, or refill first
        if (at_leaf) {
          ++r.iter;
          closest_leaf4(r, rows, S, nt, COUNT);
          r.cur = stack.pop(r.best_t);
        }
      } else if (at_node) {
        ++r.iter;
        if (!interior4<FMA, COUNT, false>(r, stack, S, r.best_t, status, nn))
          r.cur = stack.pop(r.best_t);
      }
    }
    if (ray != kNoRay) {
      if (r.iter > icap) {
        atomicOr(status, ST_ITER);
        r.cur = kIdle;
        stack.clear();
      }
      if (r.cur == kIdle) {
        __stcs(hit + ray, make_float2(r.best_leaf < 0 ? -1.0f : r.best_t, __int_as_float(r.best_leaf)));
        ray = kNoRay;
      }
    }
  }
  if (COUNT) {
    atomicAdd(&tot->nodes, (unsigned long long)nn);
    atomicAdd(&tot->tris, (unsigned long long)nt);
  }
}

// Spatial hash of an integer cell (three large odd multipliers, xor).
__device__ __forceinline__ uint32_t photon_cell_hash(int ix, int iy, int iz, uint32_t hbits) {
  const uint32_t h = ((uint32_t)ix * 73856093u) ^ ((uint32_t)iy * 19349663u) ^ ((uint32_t)iz * 83492791u);
  return h & ((1u << hbits) - 1u);
}

// Kernel-weighted flux of the photons of one cell within distance r of x,
// weight 1 - d^2 / r^2 (Epanechnikov), added to sum.  Two records in flight.
__device__ __forceinline__ void photon_cell(const PhotonMaps& M, uint32_t map, uint2 range, float3 x, float& sum) {
  auto take = [&](float4 ph) {
    const float dx = ph.x - x.x, dy = ph.y - x.y, dz = ph.z - x.z;
    const float d2 = dx * dx + dy * dy + dz * dz;
    if (d2 < M.r2[map]) sum += ph.w * (1.0f - d2 / M.r2[map]);
  };
  for (uint32_t q = range.x; q < range.y; q += 2u) {
    const float4 a = ldg4(M.rec + q), b = ldg4(M.rec + min(q + 1u, range.y - 1u));
    take(a);
    if (q + 1u < range.y) take(b);
  }
}

// The photons of band j in map `map` around x: the (at most 8) cells of edge
// 2 r that the ball touches, duplicates of a hashed key skipped.  The ball
// spans two cells per axis: all eight ranges are read at once, then their
// records in cell order, so the chain of dependent loads is two per gather
// and one per two records, not three per cell and one per record (the bound:
// long scoreboard; closest-hit and shading stages of the camera pass 4.53 ->
// 3.73 ms with the ranges' two words as one load).  Rounding can make an axis three cells wide; those
// gathers go cell by cell.
__device__ __forceinline__ float photon_gather(const PhotonMaps& M, uint32_t map, uint32_t j, float3 x) {
  const float ic = M.inv_cell[map];
  const float r = sqrtf(M.r2[map]);
  const int lx = (int)floorf((x.x - r) * ic), hx = (int)floorf((x.x + r) * ic);
  const int ly = (int)floorf((x.y - r) * ic), hy = (int)floorf((x.y + r) * ic);
  const int lz = (int)floorf((x.z - r) * ic), hz = (int)floorf((x.z + r) * ic);
  const uint32_t base = (map * M.Bc + j) << M.hbits;
  float sum = 0.0f;
  if (hx - lx <= 1 && hy - ly <= 1 && hz - lz <= 1) {
    uint32_t key[8];
    uint2 range[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      key[c] = base | photon_cell_hash(c & 4 ? hx : lx, c & 2 ? hy : ly, c & 1 ? hz : lz, M.hbits);
      range[c] = __ldg(M.range + key[c]);
    }
#pragma unroll
    for (int c = 1; c < 8; ++c) {
      bool dup = false;
#pragma unroll
      for (int q = 0; q < c; ++q) dup |= key[q] == key[c];
      if (dup) range[c] = make_uint2(0u, 0u);
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) photon_cell(M, map, range[c], x, sum);
    return sum;
  }
  uint32_t seen[8];
  int ns = 0;
  for (int ix = lx; ix <= hx; ++ix)
    for (int iy = ly; iy <= hy; ++iy)
      for (int iz = lz; iz <= hz; ++iz) {
        const uint32_t key = base | photon_cell_hash(ix, iy, iz, M.hbits);
        bool dup = false;
        for (int q = 0; q < ns; ++q) dup |= seen[q] == key;
        if (dup || ns >= 8) continue;
        seen[ns++] = key;
        photon_cell(M, map, __ldg(M.range + key), x, sum);
      }
  return sum;
}

// Appends of a block to N queues, one atomic per queue and turn of the whole
// block: with one per warp, the half a million atomics of a wave on the same
// two or three counters bounded the shading kernels (they are served one after
// another, about one per nanosecond).  Two buffers, so that a warp
// may enter its next turn while another reads this one's.
template <int N>
struct BlockAppend {
  uint32_t first[2][N][8];  // per warp (at most 8): count, then first slot
  // All threads of the block: the slots of the queues that this thread wants.
  template <int M>
  __device__ __forceinline__ void slots(uint32_t turn, const bool (&want)[M], uint32_t* const (&counter)[M],
                                        uint32_t (&slot)[M]) {
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint32_t mask[N];
#pragma unroll
    for (int q = 0; q < N; ++q) {
      mask[q] = __ballot_sync(0xffffffffu, want[q]);
      if (lane == 0) first[turn][q][warp] = (uint32_t)__popc(mask[q]);
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (warp == (uint32_t)q % nw) {
        // lane w: warp w's count; exclusive sums over the (at most 8) warps
        const uint32_t c = lane < nw ? first[turn][q][lane] : 0u;
        uint32_t x = c;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
          if ((int)lane >= o) x += y;
        }
        uint32_t b = 0;
        const uint32_t total = __shfl_sync(0xffffffffu, x, 7);
        if (lane == 0 && total != 0u) b = atomicAdd(counter[q], total);
        b = __shfl_sync(0xffffffffu, b, 0);
        if (lane < nw) first[turn][q][lane] = b + x - c;
      }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < N; ++q) slot[q] = first[turn][q][warp] + (uint32_t)__popc(mask[q] & ((1u << lane) - 1u));
  }
};

// PM: photon-mapping camera pass -- at the first Lambertian vertex the path
// adds (rho / pi) x the photon irradiance of both maps of pm and ends (its
// sun ray, if any, finishes it).
// Latency-bound: a chain of dependent reads (ray and hit, normal and radiance,
// material row) per turn, so that resident warps count for more than the few
// spilled registers they cost, and blocks are small so that their two
// barriers per turn wait for few warps.  Two samples of the 1024 x 768 nave / one
// of two guided 1024 x 768 views of the 2M-triangle nave (shading alone):
// 3 blocks of 256 per SM, one atomic per warp and queue 47.2 / 29.2 ms; one per
// block 37.2 / 24.6; as many blocks as are resident instead of 8 per SM
// 34.8 / 23.1; 6 blocks of 128 31.8 / 21.1, 7 29.3 / 19.7, 8 28.7 / 19.4 (64
// registers), 9 28.7 / 18.9, 10 29.8 / 20.0.  Four bands (512 x 384 crystal nave, 4
// samples): 13.2 ms, then 11.5 with 3 blocks of 256, 10.3 with 4, 10.8 with 8 of 128.
// With the path's radiance touched only at vertices that add to it (waves of
// 2^24 paths): 29.0 / 19.0 -> 26.7 / 17.6 ms, four bands 10.6 -> 10.0; copying
// the next turn's ray and hit ahead (cp.async) gave half of that back.
constexpr int kShadeThreads = 128, kShadeBlocksPerSm = 8;
constexpr int kShade4Threads = 256, kShade4BlocksPerSm = 4;
template <bool RECORD, bool GUIDED, bool PM = false>
__global__ void __launch_bounds__(kShadeThreads, kShadeBlocksPerSm) k_shade(DevScene S, DevSpectra P, WaveParams w, uint32_t k,
                                               const float4* __restrict__ qin, const float2* __restrict__ hit,
                                               float4* __restrict__ qout, float4* __restrict__ sq,
                                               float* __restrict__ Lbuf, uint32_t* __restrict__ sigbuf,
                                               Counters* cnt, uint32_t cap, double* __restrict__ accum,
                                               Probe probe, uint32_t* status, GuideWave gw, PhotonMaps pm) {
  const uint32_t count = min(cnt[k].q_count, cap);
  const uint32_t stride = gridDim.x * blockDim.x;
  __shared__ BlockAppend<GUIDED ? 3 : 2> app;
  uint32_t turn = 0;
  // (every thread of the block makes the same number of turns)
  for (uint32_t base = blockIdx.x * blockDim.x; base < count; base += stride, turn ^= 1u) {
    const uint32_t i = base + threadIdx.x;
    bool emit_next = false, emit_shadow = false, emit_guide = false;
    float4 n0 = make_float4(0, 0, 0, 0), n1 = n0, s0 = n0, s1 = n0;
    float g_rho = 0.0f;
    if (i < count) {
      const float4 a = __ldcs(qin + 2 * i), b = __ldcs(qin + 2 * i + 1);
      const float2 h = __ldcs(hit + i);
      const uint32_t bits = __float_as_uint(a.w);
      const uint32_t pid = bits & kPidMask;
      const bool covered = (bits & kFlagCovered) != 0u;
      const float T = b.w;
      const float3 o = f3(a), d = f3(b);
      const PathId id = path_id(w, pid);
      const uint32_t band = w.band_first + id.j;
      // the path's radiance is read and written only where this vertex adds to
      // it or ends the path
      auto add_light = [&](float x, float y) { Lbuf[pid] = fmaf(x, y, Lbuf[pid]); };
      uint32_t sg = RECORD ? sigbuf[pid] : 0u;
      // training slot of the previous (guided) vertex: radiance gathered so far
      if (GUIDED && gw.collect != 0u && k >= 2u && k - 1u <= gw.depth && pid % gw.collect == 0u)
        ((float*)(gw.raw + kRawF4 * ((k - 2u) * gw.slots_per_vertex + pid / gw.collect) + 1u))[3] = Lbuf[pid];
      const int leaf = __float_as_int(h.y);
      bool terminate = false;
      if (leaf < 0) {
        if (RECORD) sg = mix_sig(sg, 0xFFFFFFFFu);
        if (dot(d, P.sun) >= P.cos_max) {
          if (!covered) add_light(T, __ldg(P.sunL + band));
          else if (GUIDED && (bits & kFlagGuidedEsc)) add_light(T * __ldg(P.sunL + band), gw.wesc[pid]);
        }
        terminate = true;
      } else {
        const float3 p = madd(o, h.x, d);
        const float4 nr = ldg4(S.nrm + leaf);
        const uint32_t mat = __float_as_uint(nr.w);
        if (RECORD) sg = mix_sig(sg, __float_as_uint(S.tris[3 * leaf].w));
        const float3 ng = f3(nr);
        const float3 n = dot(ng, d) < 0.0f ? ng : neg(ng);
        const float cos_i = -dot(d, n);
        const float4 m = ldg4(P.mb + mat * P.n_bands + band);
        const int type = __ldg(P.mtype + mat);
        const uint4 u = philox4x32_10(make_uint4(id.pix, id.s, band, 4u * k), w.key0, w.key1);
        if (type == 0 || type == 3) {
          if (type == 3) add_light(T, m.w);
          // next-event estimate: uniform direction in the sun cone
          const float om = u01(u.x) * P.one_minus_cos;
          const float ct = 1.0f - om;
          const float st = sqrtf(fmaxf(0.0f, om * (2.0f - om)));
          float sp_, cp_;
          sincospif(2.0f * u01(u.y), &sp_, &cp_);
          float3 t1, t2;
          onb(P.sun, t1, t2);
          const float3 wd = make_float3(st * cp_ * t1.x + st * sp_ * t2.x + ct * P.sun.x,
                                        st * cp_ * t1.y + st * sp_ * t2.y + ct * P.sun.y,
                                        st * cp_ * t1.z + st * sp_ * t2.z + ct * P.sun.z);
          const float c = dot(n, wd);
          const float3 po = madd(p, S.eps, n);
          if (c > 0.0f) {
            emit_shadow = true;
            const uint32_t fl = pid | ((PM || k == w.depth) ? kFlagTerm : 0u);
            s0 = make_float4(po.x, po.y, po.z, __uint_as_float(fl));
            s1 = make_float4(wd.x, wd.y, wd.z, T * m.z * c * __ldg(P.sunL + band) * 2.0f * P.one_minus_cos);
          }
          if (PM) {
            const float E = photon_gather(pm, 0u, id.j, p) * pm.norm[0] + photon_gather(pm, 1u, id.j, p) * pm.norm[1];
            add_light(T * m.z * (1.0f / 3.14159265358979f), E);
            terminate = true;
          } else if (k == w.depth) {
            terminate = true;
          } else if (GUIDED && k <= gw.depth) {
            // the continuation is sampled by the guide kernel (one-sample MIS)
            emit_guide = true;
            n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid | kFlagCovered));
            n1 = make_float4(n.x, n.y, n.z, T);
            g_rho = m.z;
          } else {
            // cosine-weighted continuation, weight rho
            const float rr = sqrtf(u01(u.z));
            const float zz = sqrtf(fmaxf(0.0f, 1.0f - u01(u.z)));
            float s2, c2;
            sincospif(2.0f * u01(u.w), &s2, &c2);
            float3 b1, b2;
            onb(n, b1, b2);
            const float3 nd = make_float3(rr * c2 * b1.x + rr * s2 * b2.x + zz * n.x,
                                          rr * c2 * b1.y + rr * s2 * b2.y + zz * n.y,
                                          rr * c2 * b1.z + rr * s2 * b2.z + zz * n.z);
            emit_next = true;
            n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid | kFlagCovered));
            n1 = make_float4(nd.x, nd.y, nd.z, T * m.z);
          }
        } else if (type == 1) {
          float Rs, Ts;
          thin_sheet(cos_i, m.x, m.y, __ldg(P.ad + mat * P.n_bands + band), Rs, Ts);
          if (k == w.depth) {
            terminate = true;
          } else {
            const uint4 u1 = philox4x32_10(make_uint4(id.pix, id.s, band, 4u * k + 1u), w.key0, w.key1);
            emit_next = true;
            if (u01(u1.x) < Rs / (Rs + Ts)) {
              const float3 rd = madd(d, -2.0f * dot(d, n), n);
              const float3 po = madd(p, S.eps, n);
              n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid));
              n1 = make_float4(rd.x, rd.y, rd.z, T * (Rs + Ts));
            } else {
              const float3 po = madd(p, -S.eps, n);
              n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid | (bits & (kFlagCovered | kFlagGuidedEsc))));
              n1 = make_float4(d.x, d.y, d.z, T * (Rs + Ts));
            }
          }
        } else if (type == 4) {
          // solid refracting glass (section 3 Eq. 1): a segment that ends
          // here from inside crossed the medium, Beer-Lambert with alpha =
          // 4 pi k / lambda per metre; the face reflects with the Fresnel
          // reflectance of the relative index (n entering, 1/n leaving,
          // 1 past the critical angle), else refracts by Snell's law with
          // n(lambda).  The next ray starts a short step along itself so
          // that the distance crossed inside stays exact; the step's share
          // of the attenuation is taken now.
          const bool inside = dot(ng, d) > 0.0f;
          const float alpha = __ldg(P.ad + mat * P.n_bands + band);
          float Tn = inside ? T * expf(-alpha * h.x) : T;
          if (k == w.depth) {
            terminate = true;
          } else {
            const float eta = inside ? 1.0f / m.x : m.x;
            const float R = fresnel_complex(cos_i, eta, 0.0f);
            const float r = inside ? m.x : 1.0f / m.x;
            const float kk = 1.0f - r * r * (1.0f - cos_i * cos_i);
            const uint4 u1 = philox4x32_10(make_uint4(id.pix, id.s, band, 4u * k + 1u), w.key0, w.key1);
            float3 nd;
            if (u01(u1.x) < R || kk < 0.0f) {
              nd = madd(d, -2.0f * dot(d, n), n);
            } else {
              const float3 td = madd(make_float3(r * d.x, r * d.y, r * d.z), r * cos_i - sqrtf(kk), n);
              const float il = rsqrtf(dot(td, td));
              nd = make_float3(td.x * il, td.y * il, td.z * il);
            }
            const float step = S.eps / fmaxf(fabsf(dot(nd, n)), 0.0625f);
            if (dot(nd, ng) < 0.0f) Tn *= expf(-alpha * step);
            const float3 po = madd(p, step, nd);
            emit_next = true;
            n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid));
            n1 = make_float4(nd.x, nd.y, nd.z, Tn);
          }
        } else {
          const float R = fresnel_complex(cos_i, m.x, m.y);
          if (k == w.depth) {
            terminate = true;
          } else {
            const float3 rd = madd(d, -2.0f * dot(d, n), n);
            const float3 po = madd(p, S.eps, n);
            emit_next = true;
            n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid));
            n1 = make_float4(rd.x, rd.y, rd.z, T * R);
          }
        }
      }
      if (terminate && !emit_shadow) {
        const float Lp = Lbuf[pid];
        finalize(w, id, pid, Lp, sg, Lbuf, accum, probe, RECORD);
        if (GUIDED && gw.Lfinal) gw.Lfinal[pid] = Lp;
      } else if (RECORD) {
        sigbuf[pid] = sg;
      }
    }
    const bool want[3] = {emit_next, emit_shadow, emit_guide};
    uint32_t* const counter[3] = {&cnt[k + 1].q_count, &cnt[k].s_count, &cnt[k].g_count};
    uint32_t slot[3];
    app.slots(turn, want, counter, slot);
    const uint32_t slot_n = slot[0], slot_s = slot[1];
    if (GUIDED) {
      const uint32_t slot_g = slot[2];
      if (emit_guide) {
        if (slot_g < cap) {
          gw.gq[3 * slot_g] = n0;
          gw.gq[3 * slot_g + 1] = n1;
          gw.gq[3 * slot_g + 2] =
              make_float4(g_rho, __uint_as_float(emit_shadow && slot_s < cap ? slot_s : 0xFFFFFFFFu), 0.0f, 0.0f);
        } else {
          atomicOr(status, ST_QUEUE);
        }
      }
    }
    if (emit_next) {
      if (slot_n < cap) {
        __stcs(qout + 2 * slot_n, n0);
        __stcs(qout + 2 * slot_n + 1, n1);
      } else {
        atomicOr(status, ST_QUEUE);
      }
    }
    if (emit_shadow) {
      if (slot_s < cap) {
        __stcs(sq + 2 * slot_s, s0);
        __stcs(sq + 2 * slot_s + 1, s1);
      } else {
        atomicOr(status, ST_QUEUE);
      }
    }
  }
}

// Shading for paths that carry four bands: path unit j of a pixel and
// sample carries bands band_first + j + q G, q = 0..3, G = ceil(B / 4) --
// spread over the spectrum like hero wavelengths, so that the bands of one
// path fall under different parts of the colour matching functions (four
// neighbouring bands would add their correlated noise into X, Y and Z
// almost undiluted); Philox counters are those of band j.  The bands share
// every direction until the first dispersive event:
//   Lambertian / emissive: one sun-ray direction and one cosine-sampled
//     continuation for all; per-band weights rho, emitted radiance, NEE;
//   thin glass: reflect with the mean over the carried bands of
//     R_s / (R_s + T_s), weights R_s / p or T_s / (1 - p) per band;
//   conductor: mirror, weight R per band;
//   solid glass: reflect with the mean Fresnel reflectance p, weight R / p;
//     else refraction bends each band differently, so one carried band,
//     chosen uniformly, continues with weight n_carried (1 - R) / (1 - p)
//     and the others stop (their radiance so far is kept).
// "Carried" = throughput != 0; with one band left every rule is the
// one-band rule of k_shade.  Each choice has the one-band expectation per
// band, so the four-band estimate of every band is unbiased.
template <bool RECORD>
__global__ void __launch_bounds__(kShade4Threads, kShade4BlocksPerSm) k_shade4(DevScene S, DevSpectra P, WaveParams w, uint32_t k,
                                                const float4* __restrict__ qin, const float2* __restrict__ hit,
                                                float4* __restrict__ qout, float4* __restrict__ sq,
                                                float4* __restrict__ L4, float4* __restrict__ T4,
                                                float4* __restrict__ C4, uint32_t* __restrict__ sigbuf,
                                                Counters* cnt, uint32_t cap, double* __restrict__ accum,
                                                Probe probe, uint32_t* status) {
  const uint32_t count = min(cnt[k].q_count, cap);
  const uint32_t stride = gridDim.x * blockDim.x;
  __shared__ BlockAppend<2> app;
  uint32_t turn = 0;
  for (uint32_t base = blockIdx.x * blockDim.x; base < count; base += stride, turn ^= 1u) {
    const uint32_t i = base + threadIdx.x;
    bool emit_next = false, emit_shadow = false;
    float4 n0 = make_float4(0, 0, 0, 0), n1 = n0, s0 = n0, s1 = n0;
    if (i < count) {
      const float4 a = __ldcs(qin + 2 * i), b = __ldcs(qin + 2 * i + 1);
      const float2 h = __ldcs(hit + i);
      const uint32_t bits = __float_as_uint(a.w);
      const uint32_t pid = bits & kPidMask;
      const bool covered = (bits & kFlagCovered) != 0u;
      const float3 o = f3(a), d = f3(b);
      const PathId id = path_id(w, pid);
      const uint32_t b0 = w.band_first + id.j, G = w.band_count;
      const uint32_t nv = four_band_count(w, id.j);
      const float4 t4 = T4[pid];
      float T[4] = {t4.x, t4.y, t4.z, t4.w};
      // as in k_shade, the radiances are touched only where they change
      auto add_light = [&](const float (&le)[4]) {
        const float4 l = L4[pid];
        L4[pid] = make_float4(fmaf(T[0], le[0], l.x), fmaf(T[1], le[1], l.y), fmaf(T[2], le[2], l.z), fmaf(T[3], le[3], l.w));
      };
      uint32_t sg = RECORD ? sigbuf[pid] : 0u;
      const int leaf = __float_as_int(h.y);
      bool terminate = false;
      if (leaf < 0) {
        if (RECORD) sg = mix_sig(sg, 0xFFFFFFFFu);
        if (!covered && dot(d, P.sun) >= P.cos_max) {
          float le[4];
#pragma unroll
          for (uint32_t q = 0; q < 4u; ++q) le[q] = q < nv ? __ldg(P.sunL + b0 + q * G) : 0.0f;
          add_light(le);
        }
        terminate = true;
      } else {
        const float3 p = madd(o, h.x, d);
        const float4 nr = ldg4(S.nrm + leaf);
        const uint32_t mat = __float_as_uint(nr.w);
        if (RECORD) sg = mix_sig(sg, __float_as_uint(S.tris[3 * leaf].w));
        const float3 ng = f3(nr);
        const float3 n = dot(ng, d) < 0.0f ? ng : neg(ng);
        const float cos_i = -dot(d, n);
        const uint32_t mrow = mat * P.n_bands + b0;
        // material rows of the carried bands: each branch loads only the
        // fields it reads (n, k / rho, le), which keeps fewer registers live
        const float4* mr = P.mb + mrow;
        const int type = __ldg(P.mtype + mat);
        const uint4 u = philox4x32_10(make_uint4(id.pix, id.s, b0, 4u * k), w.key0, w.key1);
        // the bands still carried (throughput != 0), else every band of the path
        uint32_t act = 0;
#pragma unroll
        for (uint32_t q = 0; q < 4u; ++q)
          if (q < nv && T[q] != 0.0f) act |= 1u << q;
        if (act == 0u) act = (1u << nv) - 1u;
        const float na = (float)__popc(act);
        if (type == 0 || type == 3) {
          float rho[4];
#pragma unroll
          for (uint32_t q = 0; q < 4u; ++q) rho[q] = q < nv ? __ldg(&mr[q * G].z) : 0.0f;
          if (type == 3) {
            float le[4];
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q) le[q] = q < nv ? __ldg(&mr[q * G].w) : 0.0f;
            add_light(le);
          }
          const float om = u01(u.x) * P.one_minus_cos;
          const float ct = 1.0f - om;
          const float st = sqrtf(fmaxf(0.0f, om * (2.0f - om)));
          float sp_, cp_;
          sincospif(2.0f * u01(u.y), &sp_, &cp_);
          float3 t1, t2;
          onb(P.sun, t1, t2);
          const float3 wd = make_float3(st * cp_ * t1.x + st * sp_ * t2.x + ct * P.sun.x,
                                        st * cp_ * t1.y + st * sp_ * t2.y + ct * P.sun.y,
                                        st * cp_ * t1.z + st * sp_ * t2.z + ct * P.sun.z);
          const float c = dot(n, wd);
          const float3 po = madd(p, S.eps, n);
          if (c > 0.0f) {
            emit_shadow = true;
            float C[4];
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q)
              C[q] = q < nv ? T[q] * rho[q] * c * __ldg(P.sunL + b0 + q * G) * 2.0f * P.one_minus_cos : 0.0f;
            C4[pid] = make_float4(C[0], C[1], C[2], C[3]);
            const uint32_t fl = pid | (k == w.depth ? kFlagTerm : 0u);
            s0 = make_float4(po.x, po.y, po.z, __uint_as_float(fl));
            s1 = make_float4(wd.x, wd.y, wd.z, 0.0f);
          }
          if (k == w.depth) {
            terminate = true;
          } else {
            const float rr = sqrtf(u01(u.z));
            const float zz = sqrtf(fmaxf(0.0f, 1.0f - u01(u.z)));
            float s2, c2;
            sincospif(2.0f * u01(u.w), &s2, &c2);
            float3 b1, b2;
            onb(n, b1, b2);
            const float3 nd = make_float3(rr * c2 * b1.x + rr * s2 * b2.x + zz * n.x,
                                          rr * c2 * b1.y + rr * s2 * b2.y + zz * n.y,
                                          rr * c2 * b1.z + rr * s2 * b2.z + zz * n.z);
#pragma unroll
            for (int q = 0; q < 4; ++q) T[q] *= rho[q];
            emit_next = true;
            n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid | kFlagCovered));
            n1 = make_float4(nd.x, nd.y, nd.z, 0.0f);
          }
        } else if (type == 1) {
          float Rs[4], Ts[4];
#pragma unroll
          for (uint32_t q = 0; q < 4u; ++q) {
            Rs[q] = 0.0f;
            Ts[q] = 1.0f;
            if (q < nv) {
              const float2 nk = __ldg((const float2*)(mr + q * G));
              thin_sheet(cos_i, nk.x, nk.y, __ldg(P.ad + mrow + q * G), Rs[q], Ts[q]);
            }
          }
          if (k == w.depth) {
            terminate = true;
          } else {
            const uint4 u1 = philox4x32_10(make_uint4(id.pix, id.s, b0, 4u * k + 1u), w.key0, w.key1);
            float pr = 0.0f;
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q)
              if (act & (1u << q)) pr += Rs[q] / (Rs[q] + Ts[q]);
            pr /= na;
            emit_next = true;
            if (u01(u1.x) < pr) {
#pragma unroll
              for (int q = 0; q < 4; ++q) T[q] *= Rs[q] / pr;
              const float3 rd = madd(d, -2.0f * dot(d, n), n);
              const float3 po = madd(p, S.eps, n);
              n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid));
              n1 = make_float4(rd.x, rd.y, rd.z, 0.0f);
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q) T[q] *= Ts[q] / (1.0f - pr);
              const float3 po = madd(p, -S.eps, n);
              n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid | (bits & kFlagCovered)));
              n1 = make_float4(d.x, d.y, d.z, 0.0f);
            }
          }
        } else if (type == 4) {
          const bool inside = dot(ng, d) > 0.0f;
          float alpha[4];
#pragma unroll
          for (uint32_t q = 0; q < 4u; ++q) alpha[q] = q < nv ? __ldg(P.ad + mrow + q * G) : 0.0f;
          if (inside) {
#pragma unroll
            for (int q = 0; q < 4; ++q) T[q] *= expf(-alpha[q] * h.x);
          }
          if (k == w.depth) {
            terminate = true;
          } else {
            float R[4], nq[4];
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q) {
              nq[q] = q < nv ? __ldg(&mr[q * G].x) : 1.0f;
              R[q] = q < nv ? fresnel_complex(cos_i, inside ? 1.0f / nq[q] : nq[q], 0.0f) : 1.0f;
            }
            const uint4 u1 = philox4x32_10(make_uint4(id.pix, id.s, b0, 4u * k + 1u), w.key0, w.key1);
            float pr = 0.0f;
#pragma unroll
            for (uint32_t q = 0; q < 4u; ++q)
              if (act & (1u << q)) pr += R[q];
            pr /= na;
            float3 nd;
            if (u01(u1.x) < pr) {
#pragma unroll
              for (int q = 0; q < 4; ++q) T[q] *= R[q] / pr;
              nd = madd(d, -2.0f * dot(d, n), n);
            } else {
              // refraction is the dispersive event: one carried band goes on
              uint32_t pick = min((uint32_t)(u01(u1.y) * na), (uint32_t)na - 1u);
              uint32_t c = 0;
#pragma unroll
              for (uint32_t q = 0; q < 4u; ++q)
                if (act & (1u << q)) {
                  if (pick == 0u) c = q;
                  pick = pick == 0u ? 0xFFFFFFFFu : pick - 1u;
                }
              float Rc = R[0], nc = nq[0];
#pragma unroll
              for (uint32_t q = 1; q < 4u; ++q)
                if (q == c) {
                  Rc = R[q];
                  nc = nq[q];
                }
              const float wgt = na * (1.0f - Rc) / (1.0f - pr);
#pragma unroll
              for (uint32_t q = 0; q < 4u; ++q) T[q] = q == c ? T[q] * wgt : 0.0f;
              const float r = inside ? nc : 1.0f / nc;
              const float kk = 1.0f - r * r * (1.0f - cos_i * cos_i);
              if (kk < 0.0f) {
                nd = madd(d, -2.0f * dot(d, n), n);  // R = 1 there: the weight is already 0
              } else {
                const float3 td = madd(make_float3(r * d.x, r * d.y, r * d.z), r * cos_i - sqrtf(kk), n);
                const float il = rsqrtf(dot(td, td));
                nd = make_float3(td.x * il, td.y * il, td.z * il);
              }
            }
            const float step = S.eps / fmaxf(fabsf(dot(nd, n)), 0.0625f);
            if (dot(nd, ng) < 0.0f) {
#pragma unroll
              for (int q = 0; q < 4; ++q) T[q] *= expf(-alpha[q] * step);
            }
            const float3 po = madd(p, step, nd);
            emit_next = true;
            n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid));
            n1 = make_float4(nd.x, nd.y, nd.z, 0.0f);
          }
        } else {
          float R[4];
#pragma unroll
          for (uint32_t q = 0; q < 4u; ++q) {
            R[q] = 0.0f;
            if (q < nv) {
              const float2 nk = __ldg((const float2*)(mr + q * G));
              R[q] = fresnel_complex(cos_i, nk.x, nk.y);
            }
          }
          if (k == w.depth) {
            terminate = true;
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) T[q] *= R[q];
            const float3 rd = madd(d, -2.0f * dot(d, n), n);
            const float3 po = madd(p, S.eps, n);
            emit_next = true;
            n0 = make_float4(po.x, po.y, po.z, __uint_as_float(pid));
            n1 = make_float4(rd.x, rd.y, rd.z, 0.0f);
          }
        }
      }
      if (terminate && !emit_shadow) {
        const float4 l4 = L4[pid];
        const float L[4] = {l4.x, l4.y, l4.z, l4.w};
        finalize4(w, id, pid, L, sg, L4, accum, probe, RECORD);
      } else if (RECORD) {
        sigbuf[pid] = sg;
      }
      if (emit_next) T4[pid] = make_float4(T[0], T[1], T[2], T[3]);
    }
    const bool want[2] = {emit_next, emit_shadow};
    uint32_t* const counter[2] = {&cnt[k + 1].q_count, &cnt[k].s_count};
    uint32_t slot[2];
    app.slots(turn, want, counter, slot);
    const uint32_t slot_n = slot[0], slot_s = slot[1];
    if (emit_next) {
      if (slot_n < cap) {
        __stcs(qout + 2 * slot_n, n0);
        __stcs(qout + 2 * slot_n + 1, n1);
      } else {
        atomicOr(status, ST_QUEUE);
      }
    }
    if (emit_shadow) {
      if (slot_s < cap) {
        __stcs(sq + 2 * slot_s, s0);
        __stcs(sq + 2 * slot_s + 1, s1);
      } else {
        atomicOr(status, ST_QUEUE);
      }
    }
  }
}

// The sun ray of path pid is finished: adds its contribution (transmittance T,
// ng sheets crossed) to the path's radiance and ends the path if it was
// waiting for it.
template <bool RECORD>
__device__ __forceinline__ void sun_ray_done(const DevSpectra& P, const WaveParams& w, uint32_t k, uint32_t bits,
                                             float contrib, float T, uint32_t ng, bool rec_sun, const GuideWave& gw,
                                             float* __restrict__ Lbuf, uint32_t* __restrict__ sigbuf,
                                             double* __restrict__ accum, const Probe& probe, float* Lfinal) {
  const uint32_t pid = bits & kPidMask;
  // an occluded ray that neither ends its path nor leaves a record changes
  // nothing (sun rays of the 1024 x 768 nave 33.6 -> 32.9 ms, four bands 5.33 -> 5.18)
  if (!RECORD && !rec_sun && !(bits & kFlagTerm) && contrib * T == 0.0f) return;
  const PathId id = path_id(w, pid);
  const float Lp = fmaf(contrib, T, Lbuf[pid]);
  if (rec_sun && pid % gw.collect == 0u)
    ((float*)(gw.raw + kRawF4 * ((k - 1u) * gw.slots_per_vertex + pid / gw.collect) + 5u))[0] =
        T * __ldg(P.sunL + w.band_first + id.j);
  uint32_t sg = 0;
  if (RECORD) sg = mix_sig(sigbuf[pid], ng);
  if (bits & kFlagTerm) {
    finalize(w, id, pid, Lp, sg, Lbuf, accum, probe, RECORD);
    if (Lfinal) Lfinal[pid] = Lp;
  } else {
    Lbuf[pid] = Lp;
    if (RECORD) sigbuf[pid] = sg;
  }
}

// The same for a path that carries four bands; its contributions wait in C4.
template <bool RECORD>
__device__ __forceinline__ void sun_ray_done4(const WaveParams& w, uint32_t bits, const float (&T)[4], uint32_t ng,
                                              float4* __restrict__ L4, const float4* __restrict__ C4,
                                              uint32_t* __restrict__ sigbuf, double* __restrict__ accum,
                                              const Probe& probe) {
  const uint32_t pid = bits & kPidMask;
  if (!RECORD && !(bits & kFlagTerm) && T[0] == 0.0f && T[1] == 0.0f && T[2] == 0.0f && T[3] == 0.0f) return;
  const float4 c4 = C4[pid], l4 = L4[pid];
  const float L[4] = {fmaf(c4.x, T[0], l4.x), fmaf(c4.y, T[1], l4.y), fmaf(c4.z, T[2], l4.z), fmaf(c4.w, T[3], l4.w)};
  uint32_t sg = 0;
  if (RECORD) sg = mix_sig(sigbuf[pid], ng);
  if (bits & kFlagTerm) {
    finalize4(w, path_id(w, pid), pid, L, sg, L4, accum, probe, RECORD);
  } else {
    L4[pid] = make_float4(L[0], L[1], L[2], L[3]);
    if (RECORD) sigbuf[pid] = sg;
  }
}

// Sun rays over the four-wide BVH (trace_variant 0, and 4 and 5, which change
// the closest-hit traversal only): the loop of k_trace4, ended by the first
// opaque hit.  NB = 4: every ray belongs to a path that carries four bands
// and gathers one transmittance per band.
template <bool RECORD, bool COUNT, int NB>
__global__ void __launch_bounds__(kTraceMaxThreads, kShadow4MinBlocks)
    k_shadow4(DevScene S, DevSpectra P, WaveParams w, uint32_t k, const float4* __restrict__ sq,
              float* __restrict__ Lbuf, uint32_t* __restrict__ sigbuf, Counters* cnt, uint32_t cap,
              double* __restrict__ accum, Probe probe, Totals* tot, uint32_t* status, int steps, int refill,
              float* Lfinal, GuideWave gw, int leaf_min, const uint32_t* __restrict__ perm, float4* __restrict__ L4,
              const float4* __restrict__ C4) {
  const bool rec_sun = gw.on && gw.collect != 0u && k <= gw.depth && k < w.depth;
  const uint32_t count = min(cnt[k].s_count, cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&tot->shadow_rays, (unsigned long long)count);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t icap = trav_cap(S);
  uint32_t nn = 0, nt = 0;
  Ray4 r;
  uint32_t local[kStack + 3];
  LocalStack stack;
  stack.local = local;
  stack.clear();
  const RayRows rows(0u);
  uint32_t ray = kNoRay, ng = 0;
  float T[NB];
#pragma unroll
  for (int q = 0; q < NB; ++q) T[q] = 1.0f;
  r.cur = kIdle;
  bool drained = count == 0u;
  for (;;) {
    const uint32_t idle = __ballot_sync(0xffffffffu, ray == kNoRay);
    if (!drained && (int)__popc(idle) >= refill) {
      const uint32_t n = __popc(idle);
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(&cnt[k].s_fetch, n);
      base = __shfl_sync(0xffffffffu, base, 0);
      if (base + n >= count) drained = true;
      const uint32_t slot = base + __popc(idle & lt);
      if (ray == kNoRay && slot < count) {
        ray = perm ? __ldg(perm + slot) : slot;
        const float4 a = __ldcs(sq + 2 * ray), b = __ldcs(sq + 2 * ray + 1);
        rows.put(kRowBits, a.w);
        rows.put(kRowContrib, b.w);
        rows.put(kRowDir, b.x);
        rows.put(kRowDir + 1, b.y);
        rows.put(kRowDir + 2, b.z);
#pragma unroll
        for (int q = 0; q < NB; ++q) T[q] = 1.0f;
        ng = 0;
        ray4_init<true>(r, rows, f3(a), f3(b));
      }
    } else if (idle == 0xffffffffu) {
      break;  // drained
    }
    // a leaf step once all but this many of the lanes with a ray have left
    // the interior (they wait at a leaf, or have finished in this round)
    const int nodes_min = (int)__popc(__ballot_sync(0xffffffffu, ray != kNoRay)) - leaf_min;
    for (int i = 0; i < steps; ++i) {
      const bool at_node = (r.cur & 7u) == 0u;
      const bool at_leaf = !at_node && r.cur != kIdle;
      const uint32_t mi = __ballot_sync(0xffffffffu, at_node);
      if (mi == 0u || (int)__popc(mi) <= nodes_min) {
        if (!__any_sync(0xffffffffu, at_leaf)) break;  // none left, or refill first
        if (at_leaf) {
          ++r.iter;
          const bool opaque = shadow_leaf4w<NB>(rows, S, P, w, r.cur >> 3, r.cur & 7u, T, ng, nt, COUNT);
          if (opaque) stack.clear();
          r.cur = stack.pop(INFINITY);
        }
      } else if (at_node) {
        ++r.iter;
        if (!interior4<true, COUNT, true>(r, stack, S, INFINITY, status, nn))
          r.cur = stack.pop(INFINITY);
      }
    }
    if (ray != kNoRay) {
      if (r.iter > icap) {
        atomicOr(status, ST_ITER);
        r.cur = kIdle;
        stack.clear();
      }
      if (r.cur == kIdle) {
        const uint32_t bits = rows.get(kRowBits);
        if constexpr (NB == 4)
          sun_ray_done4<RECORD>(w, bits, T, ng, L4, C4, sigbuf, accum, probe);
        else
          sun_ray_done<RECORD>(P, w, k, bits, rows.getf(kRowContrib), T[0], ng, rec_sun, gw, Lbuf, sigbuf, accum, probe,
                               Lfinal);
        ray = kNoRay;
      }
    }
  }
  if (COUNT) {
    atomicAdd(&tot->snodes, (unsigned long long)nn);
    atomicAdd(&tot->stris, (unsigned long long)nt);
  }
}

// Sun rays over the binary BVH (trace_variant 1-3), MODE as for k_trace.
template <bool RECORD, bool COUNT, int MODE>
__global__ void __launch_bounds__(kTraceMaxThreads, kTraceMinBlocks)
    k_shadow(DevScene S, DevSpectra P, WaveParams w, uint32_t k, const float4* __restrict__ sq,
             float* __restrict__ Lbuf, uint32_t* __restrict__ sigbuf, Counters* cnt, uint32_t cap,
             double* __restrict__ accum, Probe probe, Totals* tot, uint32_t* status, int steps, int refill,
             float* Lfinal, GuideWave gw, int leaf_min, const uint32_t* __restrict__ perm) {
  const bool rec_sun = gw.on && gw.collect != 0u && k <= gw.depth && k < w.depth;
  const uint32_t count = min(cnt[k].s_count, cap);
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd(&tot->shadow_rays, (unsigned long long)count);
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t icap = trav_cap(S);
  uint32_t nn = 0, nt = 0;
  Trav tv;
  uint2 stack[kStack];
  uint32_t ray = kNoRay, bits = 0, band = 0, ng = 0;
  float contrib = 0.0f, T = 1.0f;
  float3 dir = make_float3(0.0f, 0.0f, 0.0f);
  bool drained = count == 0u;
  for (;;) {
    const uint32_t idle = __ballot_sync(0xffffffffu, ray == kNoRay);
    if (!drained && (int)__popc(idle) >= refill) {
      const uint32_t n = __popc(idle);
      uint32_t base = 0;
      if (lane == 0) base = atomicAdd(&cnt[k].s_fetch, n);
      base = __shfl_sync(0xffffffffu, base, 0);
      if (base + n >= count) drained = true;
      if (ray == kNoRay) {
        const uint32_t slot = base + __popc(idle & lt);
        if (slot < count) {
          const uint32_t ri = perm ? __ldg(perm + slot) : slot;
          const float4 a = __ldcs(sq + 2 * ri), b = __ldcs(sq + 2 * ri + 1);
          ray = ri;
          bits = __float_as_uint(a.w);
          contrib = b.w;
          dir = f3(b);
          band = w.band_first + path_id(w, bits & kPidMask).j;
          T = 1.0f;
          ng = 0;
          if (!init_w<false, true>(tv, S, f3(a), dir)) tv.sp = -1;  // misses everything: finished
        }
      }
    }
    if (!__any_sync(0xffffffffu, ray != kNoRay)) {
      if (drained) break;
      continue;
    }
    bool done = false;
    if (MODE >= 2) {
      done = ray != kNoRay && tv.sp < 0;
      for (int i = 0; i < steps; ++i) {
        const bool act = ray != kNoRay && !done;
        const bool at_leaf = act && tv.cnt != 0u;
        const uint32_t ml = __ballot_sync(0xffffffffu, at_leaf);
        const uint32_t mi = __ballot_sync(0xffffffffu, act && !at_leaf);
        if ((ml | mi) == 0u) break;
        const bool leaf_phase = mi == 0u || (int)__popc(ml) >= leaf_min;
        if (act && at_leaf == leaf_phase) {
          if (++tv.iter > icap) {
            atomicOr(status, ST_ITER);
            done = true;
          } else if (leaf_phase) {
            done = shadow_leaf(tv.rw, S, P, dir, tv.ref, tv.cnt, band, T, ng, nt, COUNT) ||
                   !trav_pop(tv, stack, INFINITY);
          } else if (!trav_interior<true, COUNT>(tv, stack, S, INFINITY, status, nn)) {
            done = !trav_pop(tv, stack, INFINITY);
          }
        }
      }
    } else if (ray != kNoRay) {
      done = tv.sp < 0;
      for (int i = 0; i < steps && !done; ++i)
        done = shadow_step<true, COUNT, MODE == 1>(tv, stack, S, P, dir, band, T, ng, icap, status, nn, nt);
    }
    if (done) {
      sun_ray_done<RECORD>(P, w, k, bits, contrib, T, ng, rec_sun, gw, Lbuf, sigbuf, accum, probe, Lfinal);
      ray = kNoRay;
    }
  }
  if (COUNT) {
    atomicAdd(&tot->snodes, (unsigned long long)nn);
    atomicAdd(&tot->stris, (unsigned long long)nt);
  }
}

// The image's slots of one wave of whole samples: each takes its paths'
// radiances in sample order, the order and the sums of one-sample waves.
// Bound by HBM (4 bytes read per path, 16 moved per slot).
__global__ void __launch_bounds__(256) k_resolve(WaveParams w, const float* __restrict__ L,
                                                 const float4* __restrict__ L4, double* __restrict__ accum) {
  for (uint32_t r = blockIdx.x * blockDim.x + threadIdx.x; r < w.PB; r += gridDim.x * blockDim.x) {
    uint32_t pix, j;
    pixel_band(w, r, pix, j);
    if (w.nb == 4u) {
      const uint32_t nv = four_band_count(w, j);
      double* a = accum + (size_t)pix * w.B + j;
      for (uint32_t q = 0; q < nv; ++q) {
        double v = a[q * w.band_count];
        for (uint32_t s = 0; s < w.samples; ++s) {
          const float x = ((const float*)(L4 + (size_t)s * w.PB + r))[q];
          if (x != 0.0f) v += (double)x;
        }
        a[q * w.band_count] = v;
      }
    } else {
      double* a = accum + (size_t)pix * w.acc_stride + w.acc_off + j;
      double v = *a;
      for (uint32_t s = 0; s < w.samples; ++s) {
        const float x = L[(size_t)s * w.PB + r];
        if (x != 0.0f) v += (double)x;
      }
      *a = v;
    }
  }
}

// Streaming-read probe: every thread reads float4s of a buffer that fits in
// L2, `iters` passes; the sum goes to a sink so the loads are not removed.
__global__ void __launch_bounds__(512) k_l2_probe(const float4* __restrict__ buf, size_t n4, int iters,
                                                  float* __restrict__ sink) {
  float acc = 0.0f;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (int it = 0; it < iters; ++it)
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += stride) {
      const float4 v = __ldcg(buf + i);
      acc += v.x + v.y + v.z + v.w;
    }
  if (acc == 1.2345f) sink[0] = acc;
}

// ---- photon mapping (section 4) ----------------------------------------

// Photon pass: one thread per photon.  Emission from the disk tangent to the
// scene's bounding sphere on the sun's side, direction minus a uniform
// sample of the sun cone, flux L_sun cos Omega pi R_d^2 / N; then the path
// tracer's material rules, storing every Lambertian hit (direct: only
// thin-glass transmissions before it; caustic: a reflection or refraction
// before the first diffuse hit; indirect: after a diffuse hit).
__global__ void __launch_bounds__(128) k_photon_trace(DevScene S, DevSpectra P, PhotonPass pp,
                                                      float4* __restrict__ rec, uint32_t* __restrict__ keys,
                                                      uint32_t* __restrict__ vals, uint8_t* __restrict__ cls,
                                                      uint32_t* status) {
  const uint32_t total = pp.Bc * pp.N;
  for (uint32_t g = blockIdx.x * blockDim.x + threadIdx.x; g < total; g += gridDim.x * blockDim.x) {
    const uint32_t j = g / pp.N, i = g - j * pp.N;
    const uint32_t b = pp.band0 + j;
    const size_t slot0 = (size_t)g * pp.depth;
    for (uint32_t q = 0; q < pp.depth; ++q) {
      keys[slot0 + q] = kPhotonEmpty;
      vals[slot0 + q] = (uint32_t)(slot0 + q);
      rec[slot0 + q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (cls) cls[slot0 + q] = 0;
    }
    const uint4 r0 = philox4x32_10(make_uint4(i, b, 0u, 0u), pp.key0, pp.key1);
    float3 o, d;
    float phi;
    if (pp.emission == 0u) {
      const float rad = pp.Rd * sqrtf(u01(r0.x));
      float sp, cp;
      sincospif(2.0f * u01(r0.y), &sp, &cp);
      o = make_float3(pp.c0.x + rad * (cp * pp.t1.x + sp * pp.t2.x), pp.c0.y + rad * (cp * pp.t1.y + sp * pp.t2.y),
                      pp.c0.z + rad * (cp * pp.t1.z + sp * pp.t2.z));
      const float om = u01(r0.z) * P.one_minus_cos;
      const float ct = 1.0f - om;
      const float st = sqrtf(fmaxf(0.0f, om * (2.0f - om)));
      float sp2, cp2;
      sincospif(2.0f * u01(r0.w), &sp2, &cp2);
      d = make_float3(-(st * cp2 * pp.t1.x + st * sp2 * pp.t2.x + ct * P.sun.x),
                      -(st * cp2 * pp.t1.y + st * sp2 * pp.t2.y + ct * P.sun.y),
                      -(st * cp2 * pp.t1.z + st * sp2 * pp.t2.z + ct * P.sun.z));
      phi = __ldg(P.sunL + b) * ct * pp.flux;
    } else {
      // portal emission: a thin-glass triangle by its share of A |s . n|
      // (the first whose cumulative share exceeds u0), a uniform point on
      // it, a direction of the cone; nothing when the direction grazes the
      // face from behind or the way back to the sun is blocked
      const float u0 = u01(r0.x);
      uint32_t lo = 0, hi = pp.n_portal - 1u;
      while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (__ldg(pp.cdf + mid) > u0) hi = mid;
        else lo = mid + 1u;
      }
      const float4 v0 = ldg4(pp.portal + 4u * lo), v1 = ldg4(pp.portal + 4u * lo + 1u),
                   v2 = ldg4(pp.portal + 4u * lo + 2u), pn = ldg4(pp.portal + 4u * lo + 3u);
      const float su = sqrtf(u01(r0.y)), u2 = u01(r0.z);
      const float wa = 1.0f - su, wb = su * (1.0f - u2), wc = su * u2;
      const float3 pg = make_float3(wa * v0.x + wb * v1.x + wc * v2.x, wa * v0.y + wb * v1.y + wc * v2.y,
                                    wa * v0.z + wb * v1.z + wc * v2.z);
      const uint4 r1 = philox4x32_10(make_uint4(i, b, 0u, 1u), pp.key0, pp.key1);
      const float om = u01(r1.x) * P.one_minus_cos;
      const float ct = 1.0f - om;
      const float st = sqrtf(fmaxf(0.0f, om * (2.0f - om)));
      float sp2, cp2;
      sincospif(2.0f * u01(r1.y), &sp2, &cp2);
      const float3 w = make_float3(st * cp2 * pp.t1.x + st * sp2 * pp.t2.x + ct * P.sun.x,
                                   st * cp2 * pp.t1.y + st * sp2 * pp.t2.y + ct * P.sun.y,
                                   st * cp2 * pp.t1.z + st * sp2 * pp.t2.z + ct * P.sun.z);
      const float3 pnv = f3(pn);
      const float wn = dot(w, pnv);
      if (!(wn > 0.0f)) continue;
      o = madd(pg, S.eps, pnv);
      float tb;
      int lb;
      closest_hit(S, o, w, tb, lb, status);
      if (lb >= 0) continue;
      d = neg(w);
      phi = __ldg(P.sunL + b) * wn * pp.flux * pn.w;
    }
    bool nee_path = true;
    uint32_t n_diff = 0;
    for (uint32_t k = 1; k <= pp.depth; ++k) {
      float t;
      int leaf;
      closest_hit(S, o, d, t, leaf, status);
      if (leaf < 0) break;
      const float3 p = madd(o, t, d);
      const float4 nr = ldg4(S.nrm + leaf);
      const uint32_t mat = __float_as_uint(nr.w);
      const float3 ng = f3(nr);
      const float3 n = dot(ng, d) < 0.0f ? ng : neg(ng);
      const float cos_i = -dot(d, n);
      const float4 m = ldg4(P.mb + mat * P.n_bands + b);
      const int type = __ldg(P.mtype + mat);
      const uint4 u = philox4x32_10(make_uint4(i, b, 0u, 4u * k), pp.key0, pp.key1);
      if (type == 0 || type == 3) {
        const uint32_t c = n_diff > 0u ? 3u : (nee_path ? 1u : 2u);
        const size_t slot = slot0 + n_diff;
        rec[slot] = make_float4(p.x, p.y, p.z, phi);
        if (cls) cls[slot] = (uint8_t)c;
        if (c != 1u) {
          const uint32_t map = c == 2u ? 0u : 1u;
          const float ic = pp.inv_cell[map];
          const uint32_t h = photon_cell_hash((int)floorf(p.x * ic), (int)floorf(p.y * ic), (int)floorf(p.z * ic),
                                              pp.hbits);
          keys[slot] = ((map * pp.Bc + j) << pp.hbits) | h;
        }
        ++n_diff;
        if (k == pp.depth) break;
        const float rr = sqrtf(u01(u.z));
        const float zz = sqrtf(fmaxf(0.0f, 1.0f - u01(u.z)));
        float s2, c2;
        sincospif(2.0f * u01(u.w), &s2, &c2);
        float3 b1, b2;
        onb(n, b1, b2);
        d = make_float3(rr * c2 * b1.x + rr * s2 * b2.x + zz * n.x, rr * c2 * b1.y + rr * s2 * b2.y + zz * n.y,
                        rr * c2 * b1.z + rr * s2 * b2.z + zz * n.z);
        o = madd(p, S.eps, n);
        phi *= m.z;
      } else if (type == 1) {
        float Rs, Ts;
        thin_sheet(cos_i, m.x, m.y, __ldg(P.ad + mat * P.n_bands + b), Rs, Ts);
        if (k == pp.depth) break;
        const uint4 u1 = philox4x32_10(make_uint4(i, b, 0u, 4u * k + 1u), pp.key0, pp.key1);
        if (u01(u1.x) < Rs / (Rs + Ts)) {
          d = madd(d, -2.0f * dot(d, n), n);
          o = madd(p, S.eps, n);
          nee_path = false;
        } else {
          o = madd(p, -S.eps, n);
        }
        phi *= Rs + Ts;
      } else if (type == 4) {
        const bool inside = dot(ng, d) > 0.0f;
        const float alpha = __ldg(P.ad + mat * P.n_bands + b);
        if (inside) phi *= expf(-alpha * t);
        if (k == pp.depth) break;
        const float eta = inside ? 1.0f / m.x : m.x;
        const float R = fresnel_complex(cos_i, eta, 0.0f);
        const float r = inside ? m.x : 1.0f / m.x;
        const float kk = 1.0f - r * r * (1.0f - cos_i * cos_i);
        const uint4 u1 = philox4x32_10(make_uint4(i, b, 0u, 4u * k + 1u), pp.key0, pp.key1);
        if (u01(u1.x) < R || kk < 0.0f) {
          d = madd(d, -2.0f * dot(d, n), n);
        } else {
          const float3 td = madd(make_float3(r * d.x, r * d.y, r * d.z), r * cos_i - sqrtf(kk), n);
          const float il = rsqrtf(dot(td, td));
          d = make_float3(td.x * il, td.y * il, td.z * il);
        }
        const float step = S.eps / fmaxf(fabsf(dot(d, n)), 0.0625f);
        if (dot(d, ng) < 0.0f) phi *= expf(-alpha * step);
        o = madd(p, step, d);
        nee_path = false;
      } else {
        const float R = fresnel_complex(cos_i, m.x, m.y);
        if (k == pp.depth) break;
        d = madd(d, -2.0f * dot(d, n), n);
        o = madd(p, S.eps, n);
        phi *= R;
        nee_path = false;
      }
    }
  }
}

// Record range per key of the sorted photon slots, and the records in key
// order.
__global__ void k_photon_bounds(const uint32_t* __restrict__ sk, const uint32_t* __restrict__ sv, uint32_t n,
                                const float4* __restrict__ rec, float4* __restrict__ rs, uint2* __restrict__ range) {
  for (uint32_t q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const uint32_t key = sk[q];
    if (key == kPhotonEmpty) continue;
    rs[q] = rec[sv[q]];
    if (q == 0u || sk[q - 1] != key) range[key].x = q;
    if (q + 1u == n || sk[q + 1] != key) range[key].y = q + 1u;
  }
}

// ---- single-step kernels for parity tests --------------------------------

__global__ void k_philox(const uint4* __restrict__ ctr, uint4* __restrict__ out, uint64_t n, uint32_t k0, uint32_t k1) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = philox4x32_10(ctr[i], k0, k1);
}

__global__ void k_closest_rays(DevScene S, const float* __restrict__ o, const float* __restrict__ d, uint64_t n,
                               float* __restrict__ tout, int32_t* __restrict__ prim, uint32_t* status) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    float t;
    int leaf;
    closest_hit(S, make_float3(o[3 * i], o[3 * i + 1], o[3 * i + 2]), make_float3(d[3 * i], d[3 * i + 1], d[3 * i + 2]),
                t, leaf, status);
    tout[i] = leaf < 0 ? -1.0f : t;
    prim[i] = leaf < 0 ? -1 : (int32_t)__float_as_uint(S.tris[3 * leaf].w);
  }
}

__global__ void k_shadow_rays(DevScene S, DevSpectra P, const float* __restrict__ o, const float* __restrict__ d,
                              const uint32_t* __restrict__ band, uint64_t n, float* __restrict__ T,
                              uint32_t* __restrict__ ng, uint32_t* status) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t g;
    T[i] = shadow_T(S, P, make_float3(o[3 * i], o[3 * i + 1], o[3 * i + 2]), make_float3(d[3 * i], d[3 * i + 1], d[3 * i + 2]),
                    band[i], g, status);
    ng[i] = g;
  }
}

__global__ void k_optics(const float* __restrict__ c, const float* __restrict__ n, const float* __restrict__ k,
                         const float* __restrict__ lam, const float* __restrict__ dd, uint64_t count,
                         float* __restrict__ R, float* __restrict__ Rs, float* __restrict__ Ts) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count; i += (uint64_t)gridDim.x * blockDim.x) {
    R[i] = fresnel_complex(c[i], n[i], k[i]);
    if (lam != nullptr && dd != nullptr) {
      // alpha d in FP64 then rounded, as the spectra tables are prepared
      const float ad = (float)(4.0 * 3.14159265358979323846 * (double)k[i] * (double)dd[i] / ((double)lam[i] * 1e-9));
      float rs, ts;
      thin_sheet(c[i], n[i], k[i], ad, rs, ts);
      Rs[i] = rs;
      Ts[i] = ts;
    }
  }
}

int grid_for(uint64_t n, int block) {
  uint64_t g = (n + block - 1) / block;
  if (g > 65535ull * 8) g = 65535ull * 8;
  return (int)(g == 0 ? 1 : g);
}

template <bool FMA, bool COUNT, int MODE>
void trace_t(const LaunchCfg& lc, const DevScene& S, const float4* qin, const WaveBufs& b, uint32_t k,
             const uint32_t* perm, cudaStream_t st) {
  k_trace<FMA, COUNT, MODE><<<lc.grid_trace, lc.block_trace, 0, st>>>(S, qin, b.hit, b.cnt, k, b.cap, b.tot, b.status,
                                                                     lc.trace_steps, lc.trace_refill, lc.leaf_min,
                                                                     perm);
}

template <bool FMA, bool COUNT>
void trace4_t(const LaunchCfg& lc, const DevScene& S, const float4* qin, const WaveBufs& b, uint32_t k,
              const uint32_t* perm, cudaStream_t st) {
  k_trace4<FMA, COUNT><<<lc.grid_trace, lc.block_trace, trace4_smem(lc.block_trace), st>>>(S, qin, b.hit, b.cnt, k, b.cap, b.tot, b.status,
                                                                 lc.trace_steps, lc.trace_refill, lc.leaf_min, perm);
}

template <bool COUNT>
void trace_m(const LaunchCfg& lc, bool robust, const DevScene& S, const float4* qin, const WaveBufs& b, uint32_t k,
             cudaStream_t st) {
  const uint32_t* perm = (lc.sort_rays && k >= 2 && b.rperm) ? b.rperm : nullptr;
  if (lc.variant == 0) {
    if (robust) trace4_t<false, COUNT>(lc, S, qin, b, k, perm, st);
    else trace4_t<true, COUNT>(lc, S, qin, b, k, perm, st);
    return;
  }
  auto run = [&](auto fma) {
    constexpr bool F = decltype(fma)::value;
    if (lc.variant == 5) trace_t<F, COUNT, 5>(lc, S, qin, b, k, perm, st);
    else if (lc.variant == 4) trace_t<F, COUNT, 4>(lc, S, qin, b, k, perm, st);
    else if (lc.variant == 3) trace_t<F, COUNT, 2>(lc, S, qin, b, k, perm, st);
    else if (lc.variant == 2) trace_t<F, COUNT, 0>(lc, S, qin, b, k, perm, st);
    else trace_t<F, COUNT, 1>(lc, S, qin, b, k, perm, st);
  };
  if (robust) run(std::false_type{});
  else run(std::true_type{});
}

void launch_trace(const LaunchCfg& lc, bool robust, const DevScene& S, const float4* qin, const WaveBufs& b, uint32_t k,
                  cudaStream_t st) {
  if (lc.counting) trace_m<true>(lc, robust, S, qin, b, k, st);
  else trace_m<false>(lc, robust, S, qin, b, k, st);
}

template <bool RECORD, bool COUNT, int MODE>
void shadow_t(const LaunchCfg& lc, const DevScene& S, const DevSpectra& P, const WaveParams& w, uint32_t k,
              const WaveBufs& b, double* accum, const Probe& probe, float* Lfinal, const GuideWave& gw,
              cudaStream_t st) {
  const uint32_t* perm = (lc.sort_rays && b.rperm) ? b.rperm : nullptr;
  k_shadow<RECORD, COUNT, MODE><<<lc.grid_shadow, lc.block_trace, 0, st>>>(
      S, P, w, k, b.sq, b.L, b.sig, b.cnt, b.cap, accum, probe, b.tot, b.status, lc.shadow_steps, lc.shadow_refill,
      Lfinal, gw, lc.leaf_min, perm);
}

template <bool RECORD, bool COUNT, int NB>
void shadow4_t(const LaunchCfg& lc, const DevScene& S, const DevSpectra& P, const WaveParams& w, uint32_t k,
               const WaveBufs& b, double* accum, const Probe& probe, float* Lfinal, const GuideWave& gw,
               cudaStream_t st) {
  const uint32_t* perm = (lc.sort_rays && b.rperm) ? b.rperm : nullptr;
  k_shadow4<RECORD, COUNT, NB><<<lc.grid_shadow, lc.block_trace, shadow4_smem(lc.block_trace), st>>>(
      S, P, w, k, b.sq, b.L, b.sig, b.cnt, b.cap, accum, probe, b.tot, b.status, lc.shadow_steps, lc.shadow_refill,
      Lfinal, gw, lc.shadow_leaf, perm, b.L4, b.C4);
}

template <bool RECORD, bool COUNT>
void shadow_m(const LaunchCfg& lc, const DevScene& S, const DevSpectra& P, const WaveParams& w, uint32_t k,
              const WaveBufs& b, double* accum, const Probe& probe, float* Lf, const GuideWave& gw, cudaStream_t st) {
  // four bands per path: the four-wide tree (the host refuses other traversal
  // variants there)
  if (w.nb == 4u) shadow4_t<RECORD, COUNT, 4>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
  else if (lc.variant == 3) shadow_t<RECORD, COUNT, 2>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
  else if (lc.variant == 2) shadow_t<RECORD, COUNT, 0>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
  else if (lc.variant == 1) shadow_t<RECORD, COUNT, 1>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
  else shadow4_t<RECORD, COUNT, 1>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
}

void launch_shadow(const LaunchCfg& lc, const DevScene& S, const DevSpectra& P, const WaveParams& w, uint32_t k,
                   const WaveBufs& b, double* accum, const Probe& probe, float* Lf, const GuideWave& gw,
                   cudaStream_t st) {
  if (lc.record) {
    if (lc.counting) shadow_m<true, true>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
    else shadow_m<true, false>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
  } else {
    if (lc.counting) shadow_m<false, true>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
    else shadow_m<false, false>(lc, S, P, w, k, b, accum, probe, Lf, gw, st);
  }
}

template <bool SUN>
void sort_queue(const DevScene& S, const float4* q, const WaveBufs& b, uint32_t k, cudaStream_t st, int sms) {
  const int g = sms > 0 ? sms * 8 : 1024;
  cudaMemsetAsync(b.rbins, 0, kCellSortBins * sizeof(uint32_t), st);
  k_rsort_hist<SUN><<<g, 256, 0, st>>>(S, q, b.cnt, k, b.cap, b.rkey, b.rbins);
  k_cell_scan_chunks<<<kCellSortBins / 1024u, 1024, 0, st>>>(b.rbins, b.rbins + kCellSortBins);
  k_cell_scan_totals<<<1, kCellSortBins / 1024u, 0, st>>>(b.rbins + kCellSortBins);
  k_rsort_scatter<SUN><<<g, 256, 0, st>>>(b.cnt, k, b.cap, b.rkey, b.rbins, b.rperm);
}

}  // namespace

void launch_cell_scan(uint32_t* bins, cudaStream_t st) { launch_scan(bins, kCellSortBins, st); }

void launch_scan(uint32_t* data, size_t n, cudaStream_t st) {
  k_cell_scan_chunks<<<(unsigned)(n / 1024u), 1024, 0, st>>>(data, data + n);
  k_cell_scan_totals<<<1, (unsigned)(n / 1024u), 0, st>>>(data + n);
}

void launch_wave(const LaunchCfg& lcfg, const DevScene& S, const DevSpectra& P, const DevCam* cams, uint32_t n_cams,
                 const WaveParams& w, const WaveBufs& b, double* accum, const Probe& probe, cudaStream_t st,
                 int* launches, StageTimer* tm, const GuideWave* gwp, const GuideDev* gdev, const void* gpack,
                 int sms, const PhotonMaps* pm) {
  GuideWave gw{};
  if (gwp) gw = *gwp;
  const bool guided = gw.on;
  // no more blocks than the wave has paths for: a queue never holds more, and
  // a block that finds nothing still costs its start and a fetch (32 x 24 box:
  // 96 blocks instead of 1368)
  LaunchCfg lc = lcfg;
  auto blocks = [&](int block) { return (int)((w.n + (uint32_t)block - 1u) / (uint32_t)block); };
  lc.grid_trace = std::min(lc.grid_trace, blocks(lc.block_trace));
  lc.grid_shadow = std::min(lc.grid_shadow, blocks(lc.block_trace));
  // shading: as many blocks as are resident at once, each with the same share
  const int block_shade = w.nb == 4u ? kShade4Threads : kShadeThreads;
  const int grid_shade =
      std::min(lc.sms * (w.nb == 4u ? kShade4BlocksPerSm : kShadeBlocksPerSm), blocks(block_shade));
  const bool rec = lc.record;
  if (tm) tm->begin(STG_CAMERA, st);
  k_camera<<<grid_for(w.n, 256), 256, 0, st>>>(cams, n_cams, w, b.q[1], b.L, b.sig, b.cnt, rec, b.L4, b.T4, b.cap,
                                                b.status);
  if (tm) tm->end(STG_CAMERA, st);
  int nl = 1;
  for (uint32_t k = 1; k <= w.depth; ++k) {
    const float4* qin = b.q[k & 1];
    float4* qout = b.q[(k + 1) & 1];
    if (tm) tm->begin(STG_TRACE, st);
    if (lc.sort_rays && k >= 2 && b.rperm) {
      sort_queue<false>(S, qin, b, k, st, sms);
      nl += 4;
    }
    // vertex 1 starts at the cameras: where one lies outside the scene bounds,
    // the box test for any origin; later origins are surface points inside the
    // padded bounds (all closest hits of 1024 x 768 x 81 bands x 2 samples in
    // the nave: 122.2 ms, with the general test at vertex 1 124.6)
    launch_trace(lc, k == 1 && !lc.cams_inside, S, qin, b, k, st);
    if (tm) tm->end(STG_TRACE, st);
    if (tm) tm->begin(STG_SHADE, st);
    if (w.nb == 4u) {
      if (rec)
        k_shade4<true><<<grid_shade, block_shade, 0, st>>>(S, P, w, k, qin, b.hit, qout, b.sq, b.L4, b.T4, b.C4,
                                                                 b.sig, b.cnt, b.cap, accum, probe, b.status);
      else
        k_shade4<false><<<grid_shade, block_shade, 0, st>>>(S, P, w, k, qin, b.hit, qout, b.sq, b.L4, b.T4,
                                                                  b.C4, b.sig, b.cnt, b.cap, accum, probe, b.status);
    } else if (pm) {
      if (rec)
        k_shade<true, false, true><<<grid_shade, block_shade, 0, st>>>(
            S, P, w, k, qin, b.hit, qout, b.sq, b.L, b.sig, b.cnt, b.cap, accum, probe, b.status, gw, *pm);
      else
        k_shade<false, false, true><<<grid_shade, block_shade, 0, st>>>(
            S, P, w, k, qin, b.hit, qout, b.sq, b.L, b.sig, b.cnt, b.cap, accum, probe, b.status, gw, *pm);
    } else if (guided) {
      if (rec)
        k_shade<true, true><<<grid_shade, block_shade, 0, st>>>(S, P, w, k, qin, b.hit, qout, b.sq, b.L, b.sig,
                                                                     b.cnt, b.cap, accum, probe, b.status, gw, PhotonMaps{});
      else
        k_shade<false, true><<<grid_shade, block_shade, 0, st>>>(S, P, w, k, qin, b.hit, qout, b.sq, b.L, b.sig,
                                                                      b.cnt, b.cap, accum, probe, b.status, gw, PhotonMaps{});
    } else {
      if (rec)
        k_shade<true, false><<<grid_shade, block_shade, 0, st>>>(S, P, w, k, qin, b.hit, qout, b.sq, b.L, b.sig,
                                                                      b.cnt, b.cap, accum, probe, b.status, gw, PhotonMaps{});
      else
        k_shade<false, false><<<grid_shade, block_shade, 0, st>>>(S, P, w, k, qin, b.hit, qout, b.sq, b.L,
                                                                       b.sig, b.cnt, b.cap, accum, probe, b.status, gw, PhotonMaps{});
    }
    if (tm) tm->end(STG_SHADE, st);
    if (guided && k <= gw.depth && k < w.depth) {
      if (tm) tm->begin(STG_GUIDE, st);
      launch_guide_sample(*gdev, gpack, P, w, k, gw, b, accum, probe, rec, sms, st);
      if (tm) tm->end(STG_GUIDE, st);
      nl += gw.perm ? 5 : 1;  // with the query sort: histogram, 2 scans, scatter
    }
    if (tm) tm->begin(STG_SHADOW, st);
    if (lc.sort_rays && b.rperm) {
      sort_queue<true>(S, b.sq, b, k, st, sms);
      nl += 4;
    }
    launch_shadow(lc, S, P, w, k, b, accum, probe, guided ? gw.Lfinal : nullptr, gw, st);
    if (tm) tm->end(STG_SHADOW, st);
    nl += 3;
  }
  if (launches) *launches += nl;
}

void launch_resolve(const WaveParams& w, const WaveBufs& b, double* accum, int sms, cudaStream_t st) {
  const uint32_t g = std::min<uint32_t>((w.PB + 255u) / 256u, (uint32_t)(sms > 0 ? sms : 1) * 16u);
  k_resolve<<<g, 256, 0, st>>>(w, b.L, b.L4, accum);
}

void launch_photon_trace(const DevScene& S, const DevSpectra& P, const PhotonPass& pp, float4* rec, uint32_t* keys,
                         uint32_t* vals, uint8_t* cls, uint32_t* status, int sms, cudaStream_t st) {
  const uint64_t n = (uint64_t)pp.Bc * pp.N;
  const unsigned g = (unsigned)std::min<uint64_t>((n + 127) / 128, (uint64_t)(sms > 0 ? sms : 1) * 64);
  k_photon_trace<<<g, 128, trace4_smem(128), st>>>(S, P, pp, rec, keys, vals, cls, status);
}

void launch_photon_maps(const uint32_t* sorted_keys, const uint32_t* sorted_vals, uint32_t n, const float4* rec,
                        float4* rec_sorted, uint2* range, int sms, cudaStream_t st) {
  k_photon_bounds<<<(sms > 0 ? sms : 1) * 8, 256, 0, st>>>(sorted_keys, sorted_vals, n, rec, rec_sorted, range);
}

void launch_philox(const uint32_t* ctr, uint32_t* out, uint64_t n, uint32_t k0, uint32_t k1, cudaStream_t st) {
  k_philox<<<grid_for(n, 256), 256, 0, st>>>((const uint4*)ctr, (uint4*)out, n, k0, k1);
}

void launch_trace_closest_rays(const DevScene& S, const float* o, const float* d, uint64_t n, float* t, int32_t* prim,
                               uint32_t* status, cudaStream_t st) {
  k_closest_rays<<<grid_for(n, 128), 128, trace4_smem(128), st>>>(S, o, d, n, t, prim, status);
}

void launch_trace_shadow_rays(const DevScene& S, const DevSpectra& P, const float* o, const float* d,
                              const uint32_t* band, uint64_t n, float* T, uint32_t* n_glass, uint32_t* status,
                              cudaStream_t st) {
  k_shadow_rays<<<grid_for(n, 128), 128, shadow4_smem(128), st>>>(S, P, o, d, band, n, T, n_glass, status);
}

void launch_optics(const float* c, const float* n, const float* k, const float* lam, const float* d, uint64_t count,
                   float* R, float* Rs, float* Ts, cudaStream_t st) {
  k_optics<<<grid_for(count, 256), 256, 0, st>>>(c, n, k, lam, d, count, R, Rs, Ts);
}

// Orders the four children of every four-wide node by the position of
// their box centres along the sun direction s, farthest first; empty slots
// (packed reference 0) last, ties by the packed reference, so that the order
// depends only on the children and s.  Sun rays visit entered children in
// slot order and stop at the first opaque triangle: in an enclosed scene the
// occluder is most often the outer shell, which far-first order reaches
// sooner (nave: 5.2 instead of 8.0 node visits per sun ray, counted on the
// CPU).  Closest-hit traversal sorts children per ray and does not depend
// on slot order.
__global__ void k_sun_order4(uint32_t* __restrict__ nodes4, uint32_t n, float3 s) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    uint32_t* w = nodes4 + (size_t)kNode4Words * i;
    uint32_t x[kNode4Words];
#pragma unroll
    for (uint32_t q = 0; q < kNode4Words; ++q) x[q] = w[q];
    float key[4];
    uint32_t pk[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      pk[c] = x[20 + c];
      key[c] = pk[c] == 0u ? -INFINITY
                           : __uint_as_float(x[c]) * s.x + __uint_as_float(x[8 + c]) * s.y + __uint_as_float(x[16 + c]) * s.z;
    }
    int rank[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      int r = 0;
#pragma unroll
      for (int d = 0; d < 4; ++d)
        if (d != c && (key[d] > key[c] || (key[d] == key[c] && (pk[d] > pk[c] || (pk[d] == pk[c] && d < c))))) ++r;
      rank[c] = r;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
#pragma unroll
      for (int a = 0; a < 3; ++a) w[8 * a + rank[c]] = x[8 * a + c];
      w[20 + rank[c]] = x[20 + c];
      // half extents: 16-bit halves of words 4-7 (x, y) and 12-13 (z)
      uint16_t* h = (uint16_t*)w;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int at = a == 2 ? 12 : 4 + 2 * a;
        h[2 * at + rank[c]] = (uint16_t)(x[at + c / 2] >> (16 * (c & 1)));
      }
    }
  }
}

void launch_sun_order4(uint32_t* nodes4, uint32_t n, float3 sun, int sms, cudaStream_t st) {
  if (n == 0) return;
  const uint32_t grid = std::min<uint32_t>((n + 255) / 256, (uint32_t)sms * 8);
  k_sun_order4<<<grid, 256, 0, st>>>(nodes4, n, sun);
}

void launch_l2_probe(const float4* buf, size_t n4, int iters, float* sink, cudaStream_t st, int sms) {
  k_l2_probe<<<sms * 4, 512, 0, st>>>(buf, n4, iters, sink);
}

int trace_blocks_per_sm(int block) {
  int a = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_trace4<true, false>, block, trace4_smem(block));
  return a > 0 ? a : 1;
}

int shadow_blocks_per_sm(int block) {
  int a = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_shadow4<false, false, 1>, block, shadow4_smem(block));
  return a > 0 ? a : 1;
}

int num_sms(int device) {
  int v = 0;
  cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, device);
  return v;
}

}  // namespace srt
