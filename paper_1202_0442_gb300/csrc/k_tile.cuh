// k_tile.cuh -- several iterations of a small single-component lattice per
// launch (k_tile), shared by the translation units that compile it for one
// storage type each.
//
// A small lattice costs a launch per iteration, not bandwidth: 64 x 32 takes
// 2.1 us per iteration, 512^2 3.8.  Here a block reads a tile and T columns and
// rows of halo into shared memory, advances it T iterations there (the part
// that is still right shrinks by one node per side and iteration) and writes
// the tile back.  The halo is advanced redundantly by the neighbouring
// blocks, so blocks need nothing from each other within the launch.  Two
// buffers of populations, one barrier per iteration; two nodes, one above
// the other, per packed operation.
//
// What bounds it: the latency of an iteration (a pair's chain of loads,
// packed arithmetic and stores, some 300 instructions, by 16 warps): 0.7 us
// for the 64 x 32 channel, 1.2 for 256^2, besides 2 us and the loads of a
// launch.  Per iteration, against one per launch: 64 x 32 0.91 us against
// 1.84, 256^2 1.75 against 2.35, 400^2 2.87 against 3.27.  With 768 or 1024 threads
// the lattices of one round gain nothing (64 x 32, with an earlier arithmetic, 0.84
// and 1.08 us per iteration against 0.83).
#pragma once

#include "lbcollide.cuh"
#include "lbpdl.cuh"

namespace lbk {

namespace {

// one pair of nodes of a tile: columns and rows of the lattice, the
// neighbour codes (a low half: the lower node), and how many iterations
// either node can be advanced (its distance from the tile's edge)
struct TilePair {
  uint32_t codes;
  int selfa, selfb;  // slots of the two nodes in the lattice
  int flags;         // x wall (bits 0-1: 1 xlo, 2 xhi), nodes its opening holds (bits 2, 3), distance << 4,
                     // the lower node's slot in the region << 16
};

struct TileOpen {
  float m[2], b[2], r[2];  // the opening rule of the two nodes
};

// word of iteration t (as the host's step_word): the rounding dither's seed
__device__ __forceinline__ uint32_t step_seed_of(long long t) {
  uint64_t z = (uint64_t)t * 0x9e3779b97f4a7c15ULL;
  z = (z ^ (z >> 31)) * 0xbf58476d1ce4e5b9ULL;
  return (uint32_t)z | 1u;
}

// the stored value of v (in stored units) as it reads back
template <class S, int SR>
__device__ __forceinline__ void round_pair(f2 (&v)[9], uint32_t seed, int selfa, int selfb, S (&a)[9], S (&b)[9]) {
  if constexpr (sizeof(S) == 4) {
#pragma unroll
    for (int i = 0; i < 9; i++) {
      a[i] = lo(v[i]);
      b[i] = hi(v[i]);
    }
  } else {
    uint32_t pa[5], pb[5];
    if constexpr (SR == 2) {
      uint32_t ra = rnd(seed, selfa, 0, 0), rb = rnd(seed, selfb, 0, 0);
#pragma unroll
      for (int i = 0; i < 4; i++) {
        ra = ra * 1664525u + 1013904223u;
        rb = rb * 1664525u + 1013904223u;
        pa[i] = Store<S>::cvt2(lo(v[2 * i]), lo(v[2 * i + 1]), ra);
        pb[i] = Store<S>::cvt2(hi(v[2 * i]), hi(v[2 * i + 1]), rb);
      }
      ra = ra * 1664525u + 1013904223u;
      rb = rb * 1664525u + 1013904223u;
      pa[4] = Store<S>::cvt1(lo(v[8]), ra);
      pb[4] = Store<S>::cvt1(hi(v[8]), rb);
#pragma unroll
      for (int i = 0; i < 9; i++) {
        const unsigned short ua = (unsigned short)(pa[i / 2] >> (16 * (i & 1)));
        const unsigned short ub = (unsigned short)(pb[i / 2] >> (16 * (i & 1)));
        memcpy(&a[i], &ua, 2);
        memcpy(&b[i], &ub, 2);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 9; i++) {
        Store<S>::st(&a[i], 0, lo(v[i]), 1.0f);
        Store<S>::st(&b[i], 0, hi(v[i]), 1.0f);
      }
    }
#pragma unroll
    for (int i = 0; i < 9; i++) v[i] = mk2(Store<S>::ld_smem(&a[i], 0, 1.0f), Store<S>::ld_smem(&b[i], 0, 1.0f));
  }
}

template <class S, bool PM, int SR>
__global__ void __launch_bounds__(TILE_THREADS, 1) k_tile(const TileArgs t) {
  extern __shared__ float pop[];  // [2][9][TILE_NODES], then the pairs and their openings
  constexpr int PS = TILE_NODES;
  constexpr bool FOLD = Store<S>::kScaled;
  TilePair *pairs = reinterpret_cast<TilePair *>(pop + 2 * 9 * PS);
  TileOpen *opens = reinterpret_cast<TileOpen *>(pairs + PS / 2);
  dep_wait();
  const MarchLat &p = t.l;
  const int T = t.steps, W = t.tw + 2 * T, H = (t.th + 2 * T + 1) & ~1;
  const int X0 = blockIdx.x * t.tw, Y0 = blockIdx.y * t.th;  // the tile's first node
  const int np = W * (H / 2);
  const float sc = FOLD ? p.scale : 1.0f;
  const S *fin = (const S *)p.fin;
  S *fout = (S *)p.fout;
  // the region's populations and pairs
  for (int k = threadIdx.x; k < np; k += TILE_THREADS) {
    const int r = k / W, x = k - r * W, y = 2 * r;
    const int gx = wrapi(X0 - T + x, p.nx), ga = wrapi(Y0 - T + y, p.ny), gb = wrapi(Y0 - T + y + 1, p.ny);
    TilePair q;
    q.selfa = ga * p.pitch + gx;
    q.selfb = gb * p.pitch + gx;
    q.codes = (uint32_t)__ldg(p.nbc + q.selfa) | ((uint32_t)__ldg(p.nbc + q.selfb) << 16);
    const int dx = min(x, W - 1 - x);
    // of the pair: the larger of its two nodes'
    const int d = min(dx, min(y + 1, H - 1 - y));
    const int s = y * W + x;
    q.flags = min(d, 255) << 4 | s << 16;
    if (t.op.nopen && (gx == 0 || gx == p.nx - 1)) {
      TileOpen o;
      o.m[0] = o.m[1] = o.b[0] = o.b[1] = o.r[0] = o.r[1] = 0.f;
      const int row[2] = {ga, gb};
#pragma unroll 1
      for (int j = 0; j < t.op.nopen; j++) {
        const int wall = span_wall(t.op.span[j]);
        if (gx != (wall == 0 ? 0 : p.nx - 1)) continue;
#pragma unroll
        for (int n = 0; n < 2; n++) {
          if (row[n] < (t.op.span[j].wa0 >> 2) || row[n] > t.op.span[j].a1) continue;
          if (!opening_mb(t.op.span[j], t.op.rule[j], 0, row[n], p.rho_ref, sc, o.m[n], o.b[n], o.r[n]))
            continue;
          q.flags |= (wall + 1) | (4 << n);
        }
      }
      opens[k] = o;
    }
    pairs[k] = q;
#pragma unroll
    for (int i = 0; i < 9; i++) {
      pop[i * PS + s] = Store<S>::ld(fin + (size_t)i * p.plane, q.selfa, 1.0f);
      pop[i * PS + s + W] = Store<S>::ld(fin + (size_t)i * p.plane, q.selfb, 1.0f);
    }
  }
  __syncthreads();
  constexpr uint32_t NB = 0x01ef01efu, SELF = 1u << NBPOS(0, 0), SOLID = SELF | (SELF << 16);
#pragma unroll 1
  for (int n = 1; n <= T; n++) {
    const float *in = pop + ((n - 1) & 1) * 9 * PS;
    float *out = pop + (n & 1) * 9 * PS;
    const uint32_t seed = SR == 2 ? step_seed_of(t.t0 + n) : 0u;
#pragma unroll 1
    for (int k = threadIdx.x; k < np; k += TILE_THREADS) {
      const TilePair q = pairs[k];
      if (((q.flags >> 4) & 255) < n) continue;
      const bool solid = (q.codes & SOLID) == SOLID;
      if (solid && n < T) continue;
      const int s = q.flags >> 16;
      f2 v[9];
      // offsets of the lower node's sources in the row below it and of the
      // upper node's in the row above it.  The region's first and last row
      // have no such row; they are advanced with the other row of their pair
      // only, their values used nowhere, and read the row next to it instead.
      const int below = s < W ? W : 0, above = s >= (H - 2) * W ? 0 : W;
#pragma unroll
      for (int i = 0; i < 9; i++) {
        const float *a = in + i * PS + s - EY(i) * W - EX(i);
        v[i] = mk2(a[EY(i) > 0 ? below : 0], a[EY(i) < 0 ? above : W]);
      }
      if (q.codes & NB) {
        const float *a = in + s;
#pragma unroll
        for (int i = 1; i < 9; i++) {
          const uint32_t m = 1u << NBPOS(-EX(i), -EY(i));
          float va = lo(v[i]), vb = hi(v[i]);
          if (q.codes & m) va = a[OPP(i) * PS];
          if (q.codes & (m << 16)) vb = a[OPP(i) * PS + W];
          v[i] = mk2(va, vb);
        }
      }
      if (q.flags & 3) {
        const TileOpen o = opens[k];
        const f2 m = mk2(o.m[0], o.m[1]), b = mk2(o.b[0], o.b[1]), rho = mk2(o.r[0], o.r[1]);
        const bool la = q.flags & 4, lb = q.flags & 8;
        f2 h1, h5, h8;
        if ((q.flags & 3) == 1) {
          zou_he<0, sizeof(S) == 2>(v, m, b, rho, h1, h5, h8);
          v[1] = mk2(la ? lo(h1) : lo(v[1]), lb ? hi(h1) : hi(v[1]));
          v[5] = mk2(la ? lo(h5) : lo(v[5]), lb ? hi(h5) : hi(v[5]));
          v[8] = mk2(la ? lo(h8) : lo(v[8]), lb ? hi(h8) : hi(v[8]));
        } else {
          zou_he<1, sizeof(S) == 2>(v, m, b, rho, h1, h5, h8);
          v[3] = mk2(la ? lo(h1) : lo(v[3]), lb ? hi(h1) : hi(v[3]));
          v[6] = mk2(la ? lo(h5) : lo(v[6]), lb ? hi(h5) : hi(v[6]));
          v[7] = mk2(la ? lo(h8) : lo(v[7]), lb ? hi(h8) : hi(v[7]));
        }
      }
      Node1<f2> nd;
      moments1<f2, PM, FOLD>(v, p.rho_ref, p.inv_scale, nd);
      nd.Fx = vfma(nd.rho, vset<f2>(p.ax), vset<f2>(p.fx));
      nd.Fy = vfma(nd.rho, vset<f2>(p.ay), vset<f2>(p.fy));
      shift1<f2, PM, sizeof(S) == 2>(p.tau, nd);
      f2 heq[9];
      equilibrium1<f2, PM, FOLD, sizeof(S) == 2>(nd, p.scale, p.wa, p.wd, heq);
      relax<sizeof(S) == 2 ? 2 : 0>(v, heq, p.omega, p.keep);
      S a[9], b[9];
      round_pair<S, SR>(v, seed, q.selfa, q.selfb, a, b);
      if (n < T) {
#pragma unroll
        for (int i = 0; i < 9; i++) {
          out[i * PS + s] = lo(v[i]);
          out[i * PS + s + W] = hi(v[i]);
        }
        continue;
      }
      // the tile's own nodes
      const int r = k / W, lx = k - r * W - T, ly = 2 * r - T;
      if (lx < 0 || lx >= t.tw || X0 + lx >= p.nx) continue;
#pragma unroll
      for (int j = 0; j < 2; j++) {
        if (ly + j < 0 || ly + j >= t.th || Y0 + ly + j >= p.ny) continue;
        const int self = j ? q.selfb : q.selfa;
        const bool fluid = !(q.codes & (j ? SELF << 16 : SELF));
        S zero;
        Store<S>::st(&zero, 0, 0.0f, 1.0f);
#pragma unroll
        for (int i = 0; i < 9; i++) fout[(size_t)i * p.plane + self] = fluid ? (j ? b[i] : a[i]) : zero;
        if (p.fields && fluid) {
          const f2 half = vset<f2>(0.5f);
          const f2 px = vadd(nd.jx, vfma(half, nd.Fx, nd.jxl)), py = vadd(nd.jy, vfma(half, nd.Fy, nd.jyl));
          const f2 e = equilibrium_sum(heq, FOLD ? p.inv_scale : 1.0f);
          p.fields[self] = j ? hi(nd.drho) : lo(nd.drho);
          p.fields[p.plane + self] = j ? hi(px) : lo(px);
          p.fields[2 * (size_t)p.plane + self] = j ? hi(py) : lo(py);
          p.fields[3 * (size_t)p.plane + self] = j ? hi(e) : lo(e);
        }
      }
    }
    __syncthreads();
  }
}

template <class S, bool PM, int SR>
int launch_tile_p(const TileArgs &t, dim3 grid, cudaStream_t s) {
  constexpr size_t smem = 2 * 9 * TILE_NODES * 4 + TILE_NODES / 2 * (sizeof(TilePair) + sizeof(TileOpen));
  if (cudaFuncSetAttribute(k_tile<S, PM, SR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return -1;
  return launch_pdl(k_tile<S, PM, SR>, grid, dim3(TILE_THREADS), smem, s, t) == cudaSuccess ? 1 : -1;
}

template <class S, int SR>
int launch_tile_t(const TileArgs &t, dim3 grid, cudaStream_t s) {
  return t.pm ? launch_tile_p<S, true, SR>(t, grid, s) : launch_tile_p<S, false, SR>(t, grid, s);
}

}  // namespace

}  // namespace lbk
