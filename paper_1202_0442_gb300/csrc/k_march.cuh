// k_march.cuh -- two iterations of the single-component fluid lattice in
// one pass over HBM (k_march), shared by the translation units that compile
// it for one storage type each.
//
// A warp owns a strip of up to 60 columns (two x-adjacent nodes per lane;
// the first and the last lane hold the strip's halo) and walks its rows
// upward.  The populations of the rows it needs live in registers: the
// shift by one column is a shuffle with the next lane, the shift by one row
// is a row kept from the step before, and the second iteration runs one row
// behind the first on the first one's results, so that two iterations
// cost one read and one write of the lattice.  No shared memory between
// lanes and no barrier; all the arithmetic is packed, two nodes per
// instruction.
//
// What bounds it: above L2 size DRAM (porous 4096^2 FP32: 107 us per
// iteration, 5.2 TB/s under ncu; the one-iteration kernel takes 196); in L2
// the latency of a row (16 warps of 128 registers per SM): 1024^2 FP32 8.4 us
// against 11.0; in 16-bit storage issue (conversions, dithers, its longer
// arithmetic): FP16 2003 x 1501 24.4 against 33.7.  Tried on the way, with an earlier
// arithmetic (1024^2 7.8 us): the second iteration two rows behind, independent of
// the first's row (168 registers, 12 warps) 9.1 us; the rows' loop not
// unrolled (more register moves) 8.2.
#pragma once

#include "lbbatch.h"
#include "lbcollide.cuh"
#include "lbpdl.cuh"

namespace lbk {

namespace {

// two x-adjacent stored values in registers: a (low) at column x, b (high)
// at x + 1
template <class S> struct Pair;

template <> struct Pair<float> {
  using R = f2;
  static __device__ __forceinline__ R ldw(const float *p, unsigned o) {
    f2 r;
    r.v = __ldg((const unsigned long long *)(p + o));
    return r;
  }
  static __device__ __forceinline__ R ld2(const float *p, unsigned oa, unsigned ob) {
    return mk2(__ldg(p + oa), __ldg(p + ob));
  }
  // the values one column to the left / right of the pair's own
  static __device__ __forceinline__ R left(R v) { return mk2(__shfl_up_sync(0xffffffffu, hi(v), 1), lo(v)); }
  static __device__ __forceinline__ R right(R v) { return mk2(hi(v), __shfl_down_sync(0xffffffffu, lo(v), 1)); }
  // `own` where bit B of the node's code (a: low half of c, b: high half) is set
  template <int B>
  static __device__ __forceinline__ R pick(R own, R v, uint32_t c) {
    return mk2((c & (1u << B)) ? lo(own) : lo(v), (c & (1u << (16 + B))) ? hi(own) : hi(v));
  }
  static __device__ __forceinline__ R keep(R v, bool a, bool b) { return mk2(a ? lo(v) : 0.f, b ? hi(v) : 0.f); }
  static __device__ __forceinline__ f2 val(R v) { return v; }
  static __device__ __forceinline__ void st(float *p, unsigned o, R v) {
    asm volatile("st.global.b64 [%0], %1;" ::"l"(__cvta_generic_to_global(p + o)), "l"(v.v) : "memory");
  }
};

struct Pair16 {
  using R = uint32_t;
  static __device__ __forceinline__ void st32(void *p, uint32_t v) {
    asm volatile("st.global.b32 [%0], %1;" ::"l"(__cvta_generic_to_global(p)), "r"(v) : "memory");
  }
  static __device__ __forceinline__ R left(R v) {
    return __byte_perm(__shfl_up_sync(0xffffffffu, v, 1), v, 0x5432);
  }
  static __device__ __forceinline__ R right(R v) {
    return __byte_perm(v, __shfl_down_sync(0xffffffffu, v, 1), 0x5432);
  }
  template <int B>
  static __device__ __forceinline__ R pick(R own, R v, uint32_t c) {
    const uint32_t m = ((c >> B) & 0x00010001u) * 0xffffu;
    return (own & m) | (v & ~m);
  }
  static __device__ __forceinline__ R keep(R v, bool a, bool b) {
    return v & ((a ? 0xffffu : 0u) | (b ? 0xffff0000u : 0u));
  }
};

template <> struct Pair<__half> : Pair16 {
  static __device__ __forceinline__ R ldw(const __half *p, unsigned o) { return __ldg((const uint32_t *)(p + o)); }
  static __device__ __forceinline__ R ld2(const __half *p, unsigned oa, unsigned ob) {
    return (uint32_t)__ldg((const unsigned short *)(p + oa)) | ((uint32_t)__ldg((const unsigned short *)(p + ob)) << 16);
  }
  static __device__ __forceinline__ f2 val(R v) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2 *>(&v));
    return mk2(f.x, f.y);
  }
  static __device__ __forceinline__ R rn(float a, float b) {
    const __half2 h = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
  static __device__ __forceinline__ void st(__half *p, unsigned o, R v) { st32(p + o, v); }
};

template <> struct Pair<__nv_bfloat16> : Pair16 {
  static __device__ __forceinline__ R ldw(const __nv_bfloat16 *p, unsigned o) {
    return __ldg((const uint32_t *)(p + o));
  }
  static __device__ __forceinline__ R ld2(const __nv_bfloat16 *p, unsigned oa, unsigned ob) {
    return (uint32_t)__ldg((const unsigned short *)(p + oa)) | ((uint32_t)__ldg((const unsigned short *)(p + ob)) << 16);
  }
  static __device__ __forceinline__ f2 val(R v) {
    return mk2(__uint_as_float(v << 16), __uint_as_float(v & 0xffff0000u));
  }
  static __device__ __forceinline__ R rn(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&h);
  }
  static __device__ __forceinline__ void st(__nv_bfloat16 *p, unsigned o, R v) { st32(p + o, v); }
};

// the pulled populations of a row's pairs: m2, m5, m6 from the row below, z
// the row itself, p4, p7, p8 from the row above; a solid source gives back
// the node's own outgoing population (half-way bounce-back).  c: the two
// neighbour codes.  Called by whole warps.
template <class S, class R>
__device__ __forceinline__ void gather(R m2, R m5, R m6, const R (&z)[9], R p4, R p7, R p8, uint32_t c,
                                       R (&h)[9]) {
  using P = Pair<S>;
  h[0] = z[0];
  h[1] = P::left(z[1]);
  h[2] = m2;
  h[3] = P::right(z[3]);
  h[4] = p4;
  h[5] = P::left(m5);
  h[6] = P::right(m6);
  h[7] = P::right(p7);
  h[8] = P::left(p8);
  // bits of the eight neighbours of either node
  constexpr uint32_t NB = 0x01ef01efu;
  if (__any_sync(0xffffffffu, c & NB)) {
    h[1] = P::template pick<NBPOS(-1, 0)>(z[3], h[1], c);
    h[2] = P::template pick<NBPOS(0, -1)>(z[4], h[2], c);
    h[3] = P::template pick<NBPOS(1, 0)>(z[1], h[3], c);
    h[4] = P::template pick<NBPOS(0, 1)>(z[2], h[4], c);
    h[5] = P::template pick<NBPOS(-1, -1)>(z[7], h[5], c);
    h[6] = P::template pick<NBPOS(1, -1)>(z[8], h[6], c);
    h[7] = P::template pick<NBPOS(1, 1)>(z[5], h[7], c);
    h[8] = P::template pick<NBPOS(-1, 1)>(z[6], h[8], c);
  }
}

// the openings of a lane's two columns: at most one on the xlo and one on
// the xhi wall (march_ok), so each node has at most one, fixed for the
// strip.  Kept in shared memory (each lane reads its own), so that the loop
// holds no registers for it.
struct LaneOpen {
  float m[2], b[2], r[2]; // its rule (rho u_n = m S + b), 0 where there is none
  int a0[2], a1[2]; // rows it spans
  int on;           // bit 0: node a has one, 1: node b; bits 2, 3: on xhi
  int rows;         // its rule depends on the row (bit 0: a, bit 1: b)
};

__device__ __forceinline__ void lane_open(const MarchLat &p, const MarchOpen &op, const int (&x)[2], float sc, LaneOpen &L) {
  int on = 0, rows = 0;
#pragma unroll
  for (int j = 0; j < 2; j++) {
    float m = 0.f, b = 0.f, r = 0.f;
    int a0 = 1, a1 = 0;
#pragma unroll 1
    for (int k = 0; k < op.nopen; k++) {
      const int wall = span_wall(op.span[k]);
      if (x[j] != (wall == 0 ? 0 : p.nx - 1) || a0 <= a1) continue;
      if (!opening_mb(op.span[k], op.rule[k], 0, 0, p.rho_ref, sc, m, b, r)) continue;
      a0 = op.span[k].wa0 >> 2;
      a1 = op.span[k].a1;
      on |= (1 | wall << 2) << j;
      if ((op.rule[k].bits & 7) == OPEN_POISEUILLE) rows |= 1 << j;
    }
    L.m[j] = m;
    L.b[j] = b;
    L.r[j] = r;
    L.a0[j] = a0;
    L.a1[j] = a1;
  }
  L.on = on;
  L.rows = rows;
}

// the opening rules of the lane's nodes in row y
template <bool S16>
__device__ __forceinline__ void open_pair(const MarchLat &p, const MarchOpen &op, const LaneOpen &L, int y, float sc,
                                          f2 (&v)[9]) {
  const int in = L.on & ((y >= L.a0[0] && y <= L.a1[0] ? 5 : 0) | (y >= L.a0[1] && y <= L.a1[1] ? 10 : 0));
  f2 m = mk2(L.m[0], L.m[1]), b = mk2(L.b[0], L.b[1]);
  if (in & L.rows) {
    float mm[2] = {lo(m), hi(m)}, bb[2] = {lo(b), hi(b)};
#pragma unroll 1
    for (int k = 0; k < op.nopen; k++) {
      const int wall = span_wall(op.span[k]);
      float mk = 0.f, bk = 0.f, rk;
      opening_mb(op.span[k], op.rule[k], 0, y, p.rho_ref, sc, mk, bk, rk);
#pragma unroll
      for (int j = 0; j < 2; j++)
        if ((L.rows >> j & 1) && (L.on >> (2 + j) & 1) == wall) {
          mm[j] = mk;
          bb[j] = bk;
        }
    }
    m = mk2(mm[0], mm[1]);
    b = mk2(bb[0], bb[1]);
  }
  f2 l1, l5, l8, r3, r6, r7;
  const f2 rho = mk2(L.r[0], L.r[1]);
  zou_he<0, S16>(v, m, b, rho, l1, l5, l8);
  zou_he<1, S16>(v, m, b, rho, r3, r6, r7);
  const bool la = (in & 5) == 1, lb = (in & 10) == 2, ra = (in & 5) == 5, rb = (in & 10) == 10;
  v[1] = mk2(la ? lo(l1) : lo(v[1]), lb ? hi(l1) : hi(v[1]));
  v[5] = mk2(la ? lo(l5) : lo(v[5]), lb ? hi(l5) : hi(v[5]));
  v[8] = mk2(la ? lo(l8) : lo(v[8]), lb ? hi(l8) : hi(v[8]));
  v[3] = mk2(ra ? lo(r3) : lo(v[3]), rb ? hi(r3) : hi(v[3]));
  v[6] = mk2(ra ? lo(r6) : lo(v[6]), rb ? hi(r6) : hi(v[6]));
  v[7] = mk2(ra ? lo(r7) : lo(v[7]), rb ? hi(r7) : hi(v[7]));
}

// the collision of two nodes (columns xa and xb of row y), rounded to the
// storage format; the same operations as collide_store on each
template <class S, bool PM, int SR, int RX, bool OPEN, class R>
__device__ __forceinline__ void collide_pair(const MarchLat &p, const MarchOpen *op, const LaneOpen &L, int xa, int xb, int y, uint32_t seed,
                                             const R (&h)[9], R (&o)[9], f2 *fields = nullptr) {
  using P = Pair<S>;
  constexpr bool FOLD = Store<S>::kScaled;
  f2 v[9];
#pragma unroll
  for (int i = 0; i < 9; i++) v[i] = P::val(h[i]);
  if (OPEN) open_pair<sizeof(S) == 2>(p, *op, L, y, FOLD ? p.scale : 1.0f, v);
  Node1<f2> n;
  moments1<f2, PM, FOLD>(v, p.rho_ref, p.inv_scale, n);
  n.Fx = vfma(n.rho, vset<f2>(p.ax), vset<f2>(p.fx));
  n.Fy = vfma(n.rho, vset<f2>(p.ay), vset<f2>(p.fy));
  shift1<f2, PM, sizeof(S) == 2>(p.tau, n);
  f2 heq[9];
  equilibrium1<f2, PM, FOLD, sizeof(S) == 2>(n, p.scale, p.wa, p.wd, heq);
  if (fields) {
    const f2 half = vset<f2>(0.5f);
    fields[0] = n.drho;
    fields[1] = vadd(n.jx, vfma(half, n.Fx, n.jxl));
    fields[2] = vadd(n.jy, vfma(half, n.Fy, n.jyl));
    fields[3] = equilibrium_sum(heq, FOLD ? p.inv_scale : 1.0f);
  }
  relax<sizeof(S) == 2 ? 2 : RX>(v, heq, p.omega, p.keep);
  if constexpr (sizeof(S) == 4) {
#pragma unroll
    for (int i = 0; i < 9; i++) o[i] = v[i];
  } else if constexpr (SR == 2) {
    // the dithers of collide_store: a hash per node, one step of a linear
    // congruential sequence per two directions
    uint32_t ra = rnd(seed, y * p.pitch + xa, 0, 0), rb = rnd(seed, y * p.pitch + xb, 0, 0);
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      ra = ra * 1664525u + 1013904223u;
      rb = rb * 1664525u + 1013904223u;
      const uint32_t a = Store<S>::cvt2(lo(v[i]), lo(v[i + 1]), ra);
      const uint32_t b = Store<S>::cvt2(hi(v[i]), hi(v[i + 1]), rb);
      o[i] = __byte_perm(a, b, 0x5410);
      o[i + 1] = __byte_perm(a, b, 0x7632);
    }
    ra = ra * 1664525u + 1013904223u;
    rb = rb * 1664525u + 1013904223u;
    o[8] = Store<S>::cvt1(lo(v[8]), ra) | (Store<S>::cvt1(hi(v[8]), rb) << 16);
  } else {
#pragma unroll
    for (int i = 0; i < 9; i++) o[i] = P::rn(lo(v[i]), hi(v[i]));
  }
}

// two iterations of rows [ys, ye) of the columns [X0, X1), by one
// warp; OPEN: the strip's columns or their halo touch a wall with openings
template <class S, bool PM, int SR, int RX, bool FIELDS, bool OPEN, int U>
__device__ __forceinline__ void march_strip(const MarchLat &p, const MarchOpen *op, LaneOpen *lanes, int X0, int X1,
                                            int ys, int ye) {
  using P = Pair<S>;
  using R = typename P::R;
  const int lane = threadIdx.x;
  const int xa = X0 - 2 + 2 * lane;  // the lane's columns xa, xa + 1
  // wrapped columns; lanes past the strip's halo repeat its last pair
  const int xc = min(xa, (X1 + 1) & ~1);
  const int wa = wrapi(xc, p.nx), wb = wrapi(xc + 1, p.nx);
  const bool wide = __all_sync(0xffffffffu, !(wa & 1) && wb == wa + 1);
  LaneOpen &L = lanes[OPEN ? threadIdx.y * 32 + lane : 0];
  if (OPEN) lane_open(p, *op, {wa, wb}, Store<S>::kScaled ? p.scale : 1.0f, L);
  const bool mine = xa >= X0 && xa < X1;
  const bool bcol = xa + 1 < X1;  // an odd lattice's last pair ends in row padding
  // lanes that share the lane's 32-byte sector
  constexpr int LPS = 16 / (int)sizeof(S);
  const int gs = lane - ((xa >> 1) & (LPS - 1));
  constexpr unsigned GM = (1u << LPS) - 1u;
  const unsigned sector = gs >= 0 ? GM << gs : GM >> -gs;
  const unsigned Pl = p.plane;
  const S *fin = (const S *)p.fin;
  S *fout = (S *)p.fout;

  auto load = [&](int row, R(&v)[9], uint32_t &c) {
    const unsigned ro = (unsigned)row * (unsigned)p.pitch;
    const unsigned oa = ro + wa, ob = ro + wb;
    if (wide) {
      c = __ldg((const uint32_t *)(p.nbc + oa));
#pragma unroll
      for (int i = 0; i < 9; i++) v[i] = P::ldw(fin + (size_t)i * Pl, oa);
    } else {
      c = (uint32_t)__ldg(p.nbc + oa) | ((uint32_t)__ldg(p.nbc + ob) << 16);
#pragma unroll
      for (int i = 0; i < 9; i++) v[i] = P::ld2(fin + (size_t)i * Pl, oa, ob);
    }
  };
  auto store = [&](int row, const R(&v)[9], uint32_t c) {
    constexpr uint32_t SELF = 1u << NBPOS(0, 0);
    const bool fa = mine && !(c & SELF), fb = mine && bcol && !(c & (SELF << 16));
    const unsigned busy = __ballot_sync(0xffffffffu, fa || fb);
    const unsigned o = (unsigned)row * (unsigned)p.pitch + (unsigned)xa;
    if (mine && (busy & sector)) {
      if (fa && fb) {
#pragma unroll
        for (int i = 0; i < 9; i++) P::st(fout + (size_t)i * Pl, o, v[i]);
      } else {
        // solid nodes hold zeros (in sectors with a fluid node)
#pragma unroll
        for (int i = 0; i < 9; i++) P::st(fout + (size_t)i * Pl, o, P::keep(v[i], fa, fb));
      }
    }
  };
  auto next = [&](int y) { return y + 1 == p.ny ? 0 : y + 1; };

  R z[9], q[9], h[9], m2, m5, m6;
  uint32_t cz, cq, cl = 0;
  int yz = wrapi(ys - 2, p.ny);
  load(yz, z, cz);
  m2 = z[2];
  m5 = z[5];
  m6 = z[6];
  yz = next(yz);
  load(yz, z, cz);
  int yq = next(yz);
  load(yq, q, cq);
  // second iteration: the row below (s2, s5, s6) and the row itself
  R s2 = m2, s5 = m5, s6 = m6, s[9];
#pragma unroll
  for (int i = 0; i < 9; i++) s[i] = z[i];
#pragma unroll U
  for (int k = ys - 1; k <= ye; k++) {
    gather<S>(m2, m5, m6, z, q[4], q[7], q[8], cz, h);
    const uint32_t c = cz;
    const int y = yz;
    m2 = z[2];
    m5 = z[5];
    m6 = z[6];
#pragma unroll
    for (int i = 0; i < 9; i++) z[i] = q[i];
    cz = cq;
    yz = yq;
    yq = next(yq);
    if (k < ye) load(yq, q, cq);
    R o[9];
    collide_pair<S, PM, SR, RX, OPEN>(p, op, L, wa, wb, y, p.seed, h, o);
    if (k > ys) {
      // the second iteration of row k - 1
      const int y2 = k - 1;
      R h2[9], o2[9];
      f2 fl[NFIELD];
      gather<S>(s2, s5, s6, s, o[4], o[7], o[8], cl, h2);
      collide_pair<S, PM, SR, RX, OPEN>(p, op, L, wa, wb, y2, p.seed2, h2, o2, FIELDS ? fl : nullptr);
      store(y2, o2, cl);
      if (FIELDS) {
        constexpr uint32_t SELF = 1u << NBPOS(0, 0);
        const unsigned at = (unsigned)y2 * (unsigned)p.pitch + (unsigned)xa;
#pragma unroll
        for (int i = 0; i < NFIELD; i++) {
          if (mine && !(cl & SELF)) p.fields[(size_t)i * Pl + at] = lo(fl[i]);
          if (mine && bcol && !(cl & (SELF << 16))) p.fields[(size_t)i * Pl + at + 1] = hi(fl[i]);
        }
      }
    }
    s2 = s[2];
    s5 = s[5];
    s6 = s[6];
#pragma unroll
    for (int i = 0; i < 9; i++) s[i] = o[i];
    cl = c;
  }
}

// One strip and one segment of rows per warp.  The border strips of a
// lattice with openings come first (a row of theirs takes longer) and take
// their own copy of the loop, so that the others carry neither the
// registers nor the instructions of the opening rules.
template <class S, bool PM, int SR, int RX, bool FIELDS>
__global__ void __launch_bounds__(128, 4) k_march(const MarchArgs a) {
  __shared__ LaneOpen lanes[128];
  dep_wait();
  const MarchLat &g = a.l;
  const int b = (int)blockIdx.x - a.eb;
  if (b < 0) {
    const int e = blockIdx.x * blockDim.y + threadIdx.y;
    const int X0 = (e & 1) * a.last, ys = (e >> 1) * a.eseg;
    if (ys < g.ny && !((e & 1) && a.last == 0))
      march_strip<S, PM, SR, RX, FIELDS, true, 1>(a.l, &a.op, lanes, X0, min(X0 + a.sw, g.nx), ys, min(ys + a.eseg, g.ny));
  } else {
    const int row = b / a.bx, strip = (b - row * a.bx) * blockDim.y + threadIdx.y;
    if (strip < a.strips) {
      const int X0 = a.x0 + strip * a.sw, ys = row * a.seg;
      march_strip<S, PM, SR, RX, FIELDS, false, 2>(a.l, &a.op, lanes, X0, min(X0 + a.sw, g.nx), ys, min(ys + a.seg, g.ny));
    }
  }
}

// the same for the lattices of a batch: a task per warp, the lattice's
// parameters in shared memory.  The loop is not unrolled: with them in
// general registers the unrolled copy spills 188 B instead of 60 (256
// lattices FP32, with an earlier arithmetic, 200 us per iteration against 192).
// 256 lattices with exact momentum: 178 us per iteration, k_batch, at 72 B per
// node and iteration, 270.  The launch numbers of its two iterations are
// those of k_batch (tick), so the dithers do not depend on which of the two
// kernels advances an iteration.
template <class S, bool PM, int SR>
__global__ void __launch_bounds__(128, 4) k_march_batch(const MarchBatch b, int parity) {
  __shared__ MarchBatchLat lats[4];
  const unsigned int launch_no = b.tick[parity];
  if (blockIdx.x == 0 && threadIdx.x == 0 && threadIdx.y == 0) {
    b.tick[1 - parity] = launch_no + 2u;
    b.counters[1 - parity] = 0;
  }
  const int k = blockIdx.x * 4 + threadIdx.y;
  if (k >= b.ntasks) return;
  const int4 t = __ldg(b.tasks + k);
  MarchBatchLat &m = lats[threadIdx.y];
  static_assert(sizeof(MarchBatchLat) % 4 == 0 && sizeof(MarchBatchLat) <= 128 + 32, "two words per lane");
  const uint32_t *src = reinterpret_cast<const uint32_t *>(b.lat + t.x);
  for (int i = threadIdx.x; i < (int)(sizeof(MarchBatchLat) / 4); i += 32) reinterpret_cast<uint32_t *>(&m)[i] = __ldg(src + i);
  __syncwarp();
  if (threadIdx.x == 0) {
    m.l.seed = mix32(launch_no * 0x9e3779b9u + (uint32_t)t.x);
    m.l.seed2 = mix32((launch_no + 1u) * 0x9e3779b9u + (uint32_t)t.x);
  }
  __syncwarp();
  march_strip<S, PM, SR, 0, false, false, 1>(m.l, nullptr, nullptr, t.y, min(t.y + m.sw, m.l.nx), t.z,
                                             min(t.z + t.w, m.l.ny));
}

template <class S, int SR>
int launch_march_batch_t(const MarchBatch &b, int parity, cudaStream_t s) {
  const dim3 grid((b.ntasks + 3) / 4), block(32, 4);
  if (b.pm) k_march_batch<S, true, SR><<<grid, block, 0, s>>>(b, parity);
  else k_march_batch<S, false, SR><<<grid, block, 0, s>>>(b, parity);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

template <class S, int SR, int RX>
int launch_march_r(const MarchArgs &a, dim3 grid, dim3 block, cudaStream_t s) {
  cudaError_t e;
  if (a.l.fields)
    e = a.pm ? launch_pdl(k_march<S, true, SR, RX, true>, grid, block, 0, s, a)
               : launch_pdl(k_march<S, false, SR, RX, true>, grid, block, 0, s, a);
  else
    e = a.pm ? launch_pdl(k_march<S, true, SR, RX, false>, grid, block, 0, s, a)
               : launch_pdl(k_march<S, false, SR, RX, false>, grid, block, 0, s, a);
  return e == cudaSuccess ? 1 : -1;
}

template <class S, int SR>
int launch_march_t(const MarchArgs &a, dim3 grid, dim3 block, cudaStream_t s) {
  if constexpr (sizeof(S) == 2) return launch_march_r<S, SR, 2>(a, grid, block, s);
  else return a.l.omega >= 1.0f ? launch_march_r<S, SR, 1>(a, grid, block, s) : launch_march_r<S, SR, 2>(a, grid, block, s);
}

}  // namespace

}  // namespace lbk
