// The derivative pass of FP64 patches whose edge is known at compile time
// (6, 9, 12), by some or all threads of a block. As derive_patch (derive.cuh),
// with the order of work that the fixed edge allows: a value is converted as it
// is gathered; the first derivatives along y and z that the mixed ones are taken
// from are those of the points' own sums, kept in shared memory (Ey widened
// along x, Ez along x and y), and only the widened rim is taken for them alone;
// the mixed derivatives are integer sums too.
//
// What bounds it: instruction issue and the latency of its phases (three
// barriers a field; ncu, 1000 patches of 9^3: 0.78 ms, issue slots 52 % busy, the
// integer pipe 65 %). 22 k thread instructions a point, 91 on the FP64 pipe (33
// without the conversions; the general pass has 286 for the sums of 14 fields and
// all mixed derivatives), so that it can run beside the algebra, which needs all of
// that pipe (stage_pair.cuh). As a launch of its own it took, against the
// general pass, one RK4 step of 140 patches of 12^3 from 3.51 to 3.36 ms, of 1000
// patches of 6^3 from 3.56 to 3.09 ms; with 9^3 patches, where the general pass
// has a fixed edge too, the two were within 3 % of one another either way.
#pragma once

#include "derive.cuh"

namespace ccz4 {

namespace {

// First-derivative sum along stride s of FP64 values in shared memory, none of them wild (ANY: of any values).
template <bool ANY>
__device__ __forceinline__ double first_of(const double *e, int s) {
  if constexpr (ANY) return fx_first(e[s], e[-s], e[2 * s], e[-2 * s]);
  else return fx_first_in(e[s], e[-s], e[2 * s], e[-2 * s]);
}

// A barrier of the THREADS threads (whole warps) that share barrier `bar`.
template <int THREADS>
__device__ __forceinline__ void block_sync(int bar) {
  asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(THREADS) : "memory");
}

// The same, and whether `mine` holds on any of them.
template <int THREADS>
__device__ __forceinline__ bool block_any(int bar, bool mine) {
  unsigned any;
  asm volatile("{ .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.or.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q; }"
               : "=r"(any) : "r"((unsigned)mine), "r"(bar), "n"(THREADS) : "memory");
  return any != 0;
}

// Source of every tile point of patch n (single level: looked up here; mesh:
// the host's table), and a mesh patch's interpolations entry by entry where
// the host planned no separable tables (into the tile buffer).
template <int SRC, int THREADS, int PF>
__device__ __forceinline__ void derive_sources(const GridView &g, const double *__restrict__ src, double *tile,
                                               const FieldList &fl, int n, int group, int groups, int *idx, int tid) {
  const int p = PF > 0 ? PF : g.p, T = PF > 0 ? PF + 2 * HALO : g.T, T3 = PF > 0 ? T * T * T : (int)g.T3;
  if (SRC == FROM_MESH) {
    const int *sp = g.src + (long long)n * T3;
    for (int t = tid; t < T3; t += THREADS) idx[t] = __ldg(sp + t);
    if (__ldg(g.xbeg + n + 1) > __ldg(g.xbeg + n)) return;
    const int e1 = __ldg(g.ibeg + n + 1);
    for (int e = __ldg(g.ibeg + n) + tid; e < e1; e += THREADS) {
      const InterpEntry *ep = g.interp + e;
      int c[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) c[k] = __ldg(&ep->src[k]);
      const int r = __ldg(&ep->r), t = __ldg(&ep->t);
      for (int j = group; j < fl.n; j += groups) {
        const int v = fl.f[j];
        __stcs(tile + ((long long)v * g.n_patches + n) * T3 + t,
               interp_value(c, r & 3, (r >> 2) & 3, (r >> 4) & 3, src + v * g.S));
      }
    }
  } else if (SRC == FROM_LEVEL) {
    const int bx = __ldg(g.ijk + 3 * n) * p - HALO;
    const int by = __ldg(g.ijk + 3 * n + 1) * p - HALO;
    const int bz = __ldg(g.ijk + 3 * n + 2) * p - HALO;
    for (int t = tid; t < T3; t += THREADS) {
      const int lz = t / (T * T), ly = (t / T) % T, lx = t % T;
      idx[t] = (int)locate(g, bx + lx, by + ly, bz + lz);
    }
  }
}

// The separable interpolations of a mesh patch's field (see XJob) into its
// tile, through scratch of nx + ny values; ends with a barrier.
template <int THREADS>
__device__ __forceinline__ void derive_interpolate(const GridView &g, const double *__restrict__ sv, double *tv, int n,
                                                   double *scratch, int tid, int bar) {
  constexpr int JM = (1 << JOB_BITS) - 1;
  const int xb0 = __ldg(g.xbeg + n), nx = __ldg(g.xbeg + n + 1) - xb0;
  if (nx == 0) return;
  const int yb0 = __ldg(g.ybeg + n), ny = __ldg(g.ybeg + n + 1) - yb0, e0 = __ldg(g.ibeg + n), e1 = __ldg(g.ibeg + n + 1);
  double *xv = scratch, *yv = scratch + nx;
  for (int q = tid; q < nx; q += THREADS) {
    const XJob *J = g.xjob + xb0 + q;
    const int rx = __ldg(&J->rx);
    const double q0 = __ldg(sv + __ldg(&J->s0));
    xv[q] = rx ? lerp3(rx, q0, __ldg(sv + __ldg(&J->s1))) : q0;
  }
  block_sync<THREADS>(bar);
  for (int q = tid; q < ny; q += THREADS) {
    const int k = __ldg(g.yjob + yb0 + q);
    yv[q] = lerp3((k >> (2 * JOB_BITS)) & 3, xv[k & JM], xv[(k >> JOB_BITS) & JM]);
  }
  block_sync<THREADS>(bar);
  for (int e = e0 + tid; e < e1; e += THREADS) {
    const int k = __ldg(&g.zjob[e].yab);
    tv[__ldg(&g.zjob[e].t)] = lerp3((k >> (2 * JOB_BITS)) & 3, yv[k & JM], yv[(k >> JOB_BITS) & JM]);
  }
  block_sync<THREADS>(bar);
}

// ---- the pass of a patch edge known at compile time -----------------------------------
// Threads of a block and resident blocks asked for: 9^3 patches 384 threads
// (two rounds of 729 points, nine of the tile) and 68 KB, three blocks
// per SM; 12^3 patches 864 threads (two rounds) and 125 KB, one block; 6^3
// patches 224 threads (one round) and 32 KB.
template <int PF>
struct EdgeShape {
  static constexpr int threads = PF == 12 ? 864 : PF == 6 ? 224 : 384, blocks = PF == 12 ? 1 : PF == 6 ? 4 : 3;
};
constexpr int EDGE_EZ(int p) { return (p + 4) * (p + 4) * p; }
constexpr int EDGE_EY(int p) { return (p + 4) * p * p; }
// ONE: a block takes one field, whose source table then shares the place of Ez and Ey.
constexpr size_t edge_smem_bytes(int p, bool one = false) {
  const size_t T3 = (size_t)(p + 6) * (p + 6) * (p + 6);
  return 8 * (T3 + EDGE_EZ(p) + EDGE_EY(p)) + ((one ? 0 : 4 * T3) + 2 * T3 + 7) / 8 * 8;
}
static_assert(4 * 15 * 15 * 15 <= 8 * (EDGE_EZ(9) + EDGE_EY(9)), "a source table in the place of Ez and Ey");

// The fields group, group + groups, ... of the list, of patch n, into the place
// of patch `at_patch` of the derivative buffer, by the THREADS threads tid (whole
// warps) that share barrier bar. tile: the tile buffer; interpolated halo points of a mesh pass through it.
template <int SRC, int THREADS, int PF, bool CVT, bool ONE = false>
__device__ __forceinline__ void derive_edge(const GridView &g, const double *__restrict__ src, double *tile,
                                            double *__restrict__ mix, double *__restrict__ der, const LevelScale &ls,
                                            const FieldList &fl, int n, int at_patch, int group, int groups,
                                            double *smem, int tid, int bar) {
  constexpr int T = PF + 2 * HALO, T2 = T * T, T3 = T2 * T, P2 = PF * PF, P3 = P2 * PF, PE = PF + 4;
  constexpr int BATCH = (T3 + THREADS - 1) / THREADS <= 10 ? (T3 + THREADS - 1) / THREADS : 7;
  constexpr int ROUNDS = (P3 + THREADS - 1) / THREADS;
  constexpr bool MESH = SRC == FROM_MESH;
  int64_t *tw = reinterpret_cast<int64_t *>(smem);
  double *Ez = smem + T3, *Ey = Ez + EDGE_EZ(PF);
  int *idx = reinterpret_cast<int *>(ONE ? Ez : Ey + EDGE_EY(PF));
  unsigned short *ex = reinterpret_cast<unsigned short *>(ONE ? reinterpret_cast<int *>(Ey + EDGE_EY(PF)) : idx + T3);
  derive_sources<SRC, THREADS, PF>(g, src, tile, fl, n, group, groups, idx, tid);
  const int lev = MESH ? patch_level(g, n) : 0;
  const double cmix = MESH ? ls.cmix[lev] : ls.cmix[0];
  const long long pbase = (long long)n * P3, np = g.n_points;
  const long long dbase = (long long)at_patch * P3, dnp = (long long)g.wcap * P3;
  // tile offsets of this thread's points, the same for every field (few rounds: kept)
  constexpr bool KEEP = ROUNDS <= 3;
  auto tile_at = [&](int q) { return (q / P2 + HALO) * T2 + ((q / PF) % PF + HALO) * T + (q % PF + HALO); };
  auto ez_at = [&](int q) { return ((q / P2) * PE + ((q / PF) % PF + 2)) * PE + (q % PF + 2); };
  int at[KEEP ? ROUNDS : 1], az[KEEP ? ROUNDS : 1];
#pragma unroll
  for (int r = 0; r < (KEEP ? ROUNDS : 1); ++r) {
    at[r] = tile_at(tid + r * THREADS);
    az[r] = ez_at(tid + r * THREADS);
  }
  auto pick = [&](const int (&a)[KEEP ? ROUNDS : 1], int r) {
    int c = a[0];
#pragma unroll
    for (int k = 1; k < (KEEP ? ROUNDS : 1); ++k) c = r == k ? a[k] : c;
    return c;
  };
  for (int j = group; j < fl.n; j += groups) {
    const int v = fl.f[j];
    const double *sv = src + (long long)v * g.S;
    double *tv = tile + ((long long)v * g.n_patches + n) * T3;
    const int slot = mix_slot(v);
    const bool second = slot >= 0;
    block_sync<THREADS>(bar);  // the source table is written; the previous field's readers are done
    if (MESH) derive_interpolate<THREADS>(g, sv, tv, n, smem, tid, bar);
#pragma unroll 1
    for (int t0 = tid; t0 < T3; t0 += BATCH * THREADS) {
      double val[BATCH];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int t = t0 + u * THREADS;
        val[u] = 0.0;
        if (t >= T3) continue;
        const int s = idx[t];
        if (s >= 0) val[u] = __ldg(sv + s);
        else if (MESH && s <= -2) val[u] = __ldcg(tv + t);  // interpolated above (through L2)
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int t = t0 + u * THREADS;
        if (t >= T3) continue;
        unsigned e;
        tw[t] = fx_word(val[u], e);
        ex[t] = (unsigned short)e;
      }
    }
    block_sync<THREADS>(bar);
    double *d = der + 4 * v * dnp + dbase, *dp = der + (4 * NV + 3 * (second ? slot / 3 : 0)) * dnp + dbase;
    auto take = [&](auto is_second) {
      constexpr bool SECOND = decltype(is_second)::value;
      bool wild = false;  // a first derivative outside the integer range
#pragma unroll 1
      for (int r = 0; r < ROUNDS; ++r) {
        const int q = tid + r * THREADS;
        if (q >= P3) break;
        const int c = KEEP ? pick(at, r) : tile_at(q);
        double o[7];
        point_sums<SECOND, CVT>(tw + c, ex + c, T, o);
#pragma unroll
        for (int k = 0; k < 4; ++k) d[k * dnp + q] = o[k];
        if (SECOND) {
#pragma unroll
          for (int k = 0; k < 3; ++k) dp[k * dnp + q] = o[4 + k];
        }
        if (SECOND) {
          const int row = q / PF;
          Ey[row * PE + (q - row * PF + 2)] = o[1];
          Ez[KEEP ? pick(az, r) : ez_at(q)] = o[2];
          wild |= fx_wild(o[1]) | fx_wild(o[2]);
        }
      }
      if constexpr (SECOND) {
        // the rim: along z beyond the patch in x or in y (8 PF columns a plane), along y beyond it in x
        for (int h = tid; h < 8 * P2 + 4 * P2; h += THREADS) {
          const bool along_z = h < 8 * P2;
          const int k = along_z ? h : h - 8 * P2;
          const int z = k / (along_z ? 8 * PF : 4 * PF), m = k - z * (along_z ? 8 * PF : 4 * PF);
          const bool in_y = along_z && m >= 4 * PF;  // beyond the patch in y
          const int m1 = in_y ? m - 4 * PF : m, a = m1 / PF, b = m1 - a * PF;
          const int far = a < 2 ? a - 2 : PF + a - 2;  // -2, -1, PF, PF + 1
          const int x = in_y ? b : far, y = in_y ? far : b;
          const int c = (z + HALO) * T2 + (y + HALO) * T + (x + HALO);
          const double f = fx_first_sum(tw + c, ex + c, along_z ? T2 : T);
          wild |= fx_wild(f);
          if (along_z) Ez[(z * PE + (y + 2)) * PE + (x + 2)] = f;
          else Ey[(z * PF + y) * PE + (x + 2)] = f;
        }
        // the mixed derivatives; with FP64 operations at hand only where the block has need of them (they would
        // be issued for every point: 99 a point, 28.7 against 26.4 ms a step at 144^3)
        auto mixed = [&](auto any) {
#pragma unroll 1
          for (int r = 0; r < ROUNDS; ++r) {
            const int q = tid + r * THREADS;
            if (q >= P3) break;
            const int row = q / PF, z = KEEP ? pick(az, r) : ez_at(q);
            double *o = mix + (long long)slot * np + pbase + q;
            __stcs(o, first_of<decltype(any)::value>(Ey + row * PE + (q - row * PF + 2), 1) * cmix);
            __stcs(o + np, first_of<decltype(any)::value>(Ez + z, 1) * cmix);
            __stcs(o + 2 * np, first_of<decltype(any)::value>(Ez + z, PE) * cmix);
          }
        };
        if (block_any<THREADS>(bar, wild)) mixed(std::true_type());
        else mixed(std::false_type());
      }
    };
    if (second) take(std::true_type());
    else take(std::false_type());
  }
}

}  // namespace

}  // namespace ccz4
