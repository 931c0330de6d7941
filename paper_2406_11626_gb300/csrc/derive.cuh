// The derivative pass: everything a right-hand side needs of its neighbours.
//
// One block gathers a patch's halo'd tile field by field into shared memory
// and writes, for each of the patch's points, the unscaled stencil sums of
// the field: the three first-derivative sums and the Kreiss-Oliger sum, for
// the fields with second derivatives also the three pure ones, and the mixed
// second derivatives (as the halo fill forms them). The pointwise algebra
// (algebra kernels, monitors) then reads each point's values in full lines
// and touches no neighbour.
//
// Why a pass of its own: the FP64 pipe issues 2 operations per clock per SM,
// and about 45 % of the right-hand side's FP64 operations are stencil sums.
// Here they run on the integer pipes instead (fixed_stencil.cuh), at the
// occupancy and the register count of a small kernel; a value is converted
// once per tile it lands in (4.6 times at a patch edge of 9) and not once for
// each of the 19 points that read it. The algebra is left with the FP64
// operations that have to be FP64, needs no tile (nothing is reused through
// L1) and spills less.
#pragma once

#include "derive.h"
#include "fixed_stencil.cuh"
#include "halo_fill.cuh"

namespace ccz4 {

namespace {

// The stencil sums of the point at w, ex in a tile of edge T: out[0..2] first
// derivatives, out[3] dissipation, out[4..6] pure second derivatives. CVT, FIRST_CVT: as fx_point.
template <bool SECOND, bool CVT = true, bool FIRST_CVT = false, class E>
__device__ __forceinline__ void point_sums(const int64_t *w, const E *ex, int T, double *out) {
  const int st[3] = {1, T, T * T};
  fx_point<SECOND, CVT, FIRST_CVT>(w, ex, st, out);
}

// The same in FP32 from split pairs (mixed precision), whose FP32 pipe is
// wider than the integer one: first differences (hi+ - hi-) + (lo+ - lo-),
// second differences from error-free differences of the high parts (the
// reasons stand at sp_second in ccz4_algebra.cuh). On the 144^3 puncture the
// integer sums with FP32 results took the mixed step to 15.8 ms, the pairs
// to 15.3.
template <bool SECOND>
__device__ __forceinline__ void point_sums(const float2 *t, const unsigned *, int T, float *out) {
  const int st[3] = {1, T, T * T};
  const float2 c = t[0];
  float ko = 0.0f;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    float b[3], d[2];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float2 p = t[(j + 1) * st[k]], m = t[-(j + 1) * st[k]];
      float ep, em;
      const float dp = sp_two_diff<float>(p.x, c.x, ep), dm = sp_two_diff<float>(m.x, c.x, em);
      b[j] = (dp + dm) + ((ep + em) + fmaf(-2.0f, c.y, p.y + m.y));
      if (j < 2) d[j] = (p.x - m.x) + (p.y - m.y);
    }
    out[k] = fmaf(8.0f, d[0], -d[1]);
    if (SECOND) out[4 + k] = fmaf(16.0f, b[0], -b[1]);
    const float s = fmaf(15.0f, b[0], fmaf(-6.0f, b[1], b[2]));
    ko = k == 0 ? s : ko + s;
  }
  out[3] = ko;
}

// Where a patch's tile comes from: gathered through the neighbour lookup of a
// single level, or through a refined mesh's table, or read from the tile
// buffer that a halo fill has written.
enum { FROM_LEVEL = 0, FROM_MESH = 1, FROM_TILE = 2 };

// Doubles that the widened region of the mixed derivatives takes, and the
// place of the exponents with it: a field's mixed derivatives are done before
// its exponents are written, so the two share their place.
__host__ __device__ constexpr int derive_ext(int p) {
  return fill_wide(p) ? (p + 4) * (p + 4) * p : (p + 4) * p * p;
}
__host__ __device__ constexpr int derive_shared(int p) {
  const int T3 = (p + 2 * HALO) * (p + 2 * HALO) * (p + 2 * HALO), e = derive_ext(p), x = (T3 + 1) / 2;
  return e > x ? e : x;
}
// Shared memory of a block: the tile's words, the shared place above and the
// source table (not FROM_TILE). 54 KB at a patch edge of 9: four blocks per SM.
inline size_t derive_smem_bytes(int p) {
  const size_t T = (size_t)p + 2 * HALO, T3 = T * T * T;
  return T3 * (8 + 4) + 8 * (size_t)derive_shared(p);
}

// The fields group, group + groups, ... of the list, of patch n, into the place
// of patch `at_patch` of the derivative buffer, by one block of THREADS threads. NF: fields of the formulation (25, or 58 without second
// derivatives). tile: the tile buffer; interpolated halo points of a mesh pass
// through it, tile_out (FP64) has the whole tile written to it, FROM_TILE reads it.
template <int SRC, bool MIXED, int THREADS, int PF, int NF>
__device__ __forceinline__ void derive_patch(const GridView &g, const double *__restrict__ src, double *tile,
                                             double *__restrict__ mix, double *__restrict__ der, const LevelScale &ls,
                                             const FieldList &fl, int n, int at_patch, int group, int groups, bool tile_out,
                                             double *smem) {
  constexpr int BATCH = PF == 9 && THREADS == 256 ? 7 : 8;  // 15^3 tile points: two rounds of 7 x 256
  const int p = PF > 0 ? PF : g.p, T = PF > 0 ? PF + 2 * HALO : g.T;
  const int T3 = PF > 0 ? T * T * T : (int)g.T3;
  const int pe = p + 4, next = pe * p * p, p3 = p * p * p;
  const bool wide = fill_wide(p);
  double *ts = smem;
  double *ext = ts + T3;
  unsigned *ex = reinterpret_cast<unsigned *>(ext);
  int *idx = reinterpret_cast<int *>(ext + derive_shared(p));
  constexpr bool MESH = SRC == FROM_MESH;
  int e0 = 0, e1 = 0, xb0 = 0, nx = 0, yb0 = 0, ny = 0;
  if (MESH) {
    const int *sp = g.src + (long long)n * T3;
    for (int t = threadIdx.x; t < T3; t += THREADS) idx[t] = __ldg(sp + t);
    e0 = __ldg(g.ibeg + n);
    e1 = __ldg(g.ibeg + n + 1);
    xb0 = __ldg(g.xbeg + n);
    nx = __ldg(g.xbeg + n + 1) - xb0;
    yb0 = __ldg(g.ybeg + n);
    ny = __ldg(g.ybeg + n + 1) - yb0;
    // a patch without separable tables: one entry per thread, every field of the group
    for (int e = nx == 0 ? e0 + (int)threadIdx.x : e1; e < e1; e += THREADS) {
      const InterpEntry *ep = g.interp + e;
      int c[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) c[k] = __ldg(&ep->src[k]);
      const int r = __ldg(&ep->r), t = __ldg(&ep->t);
      for (int j = group; j < fl.n; j += groups) {
        const int v = fl.f[j] & ~FIELD_NO_SUMS;
        __stcs(tile + ((long long)v * g.n_patches + n) * T3 + t,
               interp_value(c, r & 3, (r >> 2) & 3, (r >> 4) & 3, src + v * g.S));
      }
    }
  } else if (SRC == FROM_LEVEL) {
    const int bx = __ldg(g.ijk + 3 * n) * p - HALO;
    const int by = __ldg(g.ijk + 3 * n + 1) * p - HALO;
    const int bz = __ldg(g.ijk + 3 * n + 2) * p - HALO;
    for (int t = threadIdx.x; t < T3; t += THREADS) {
      const int lz = t / (T * T), ly = (t / T) % T, lx = t % T;
      idx[t] = (int)locate(g, bx + lx, by + ly, bz + lz);
    }
  }
  const double cmix = MESH ? ls.cmix[patch_level(g, n)] : ls.cmix[0];
  const float cmixf = MESH ? ls.cmixf[patch_level(g, n)] : ls.cmixf[0];
  const long long pbase = (long long)n * p3, np = g.n_points;
  const long long dbase = (long long)at_patch * p3, dnp = (long long)g.wcap * p3;
  // tile offsets of this thread's points (a compile-time edge: the same for every field)
  constexpr int ROUNDS = PF > 0 ? (PF * PF * PF + THREADS - 1) / THREADS : 1;
  auto centre_at = [&](int q) {
    const int x = q % p, y = (q / p) % p, z = q / (p * p);
    return ((z + HALO) * T + (y + HALO)) * T + (x + HALO);
  };
  int at[ROUNDS];
#pragma unroll
  for (int r = 0; r < ROUNDS; ++r) at[r] = PF > 0 ? centre_at(threadIdx.x + r * THREADS) : 0;
  constexpr int JM = (1 << JOB_BITS) - 1;
  for (int j = group; j < fl.n; j += groups) {
    const int v = fl.f[j] & ~FIELD_NO_SUMS;
    const bool sums = (fl.f[j] & FIELD_NO_SUMS) == 0;
    const double *sv = src + (long long)v * g.S;
    double *tv = tile + ((long long)v * g.n_patches + n) * T3;
    const int slot = NF == NV ? mix_slot(v) : -1;
    __syncthreads();  // the source table is written; the previous field's readers are done
    if (MESH && nx > 0) {
      double *xv = ts, *yv = ts + nx;
      for (int q = threadIdx.x; q < nx; q += THREADS) {
        const XJob *J = g.xjob + xb0 + q;
        const int rx = __ldg(&J->rx);
        const double q0 = __ldg(sv + __ldg(&J->s0));
        xv[q] = rx ? lerp3(rx, q0, __ldg(sv + __ldg(&J->s1))) : q0;
      }
      __syncthreads();
      for (int q = threadIdx.x; q < ny; q += THREADS) {
        const int k = __ldg(g.yjob + yb0 + q);
        yv[q] = lerp3((k >> (2 * JOB_BITS)) & 3, xv[k & JM], xv[(k >> JOB_BITS) & JM]);
      }
      __syncthreads();
      for (int e = e0 + threadIdx.x; e < e1; e += THREADS) {
        const int k = __ldg(&g.zjob[e].yab);
        tv[__ldg(&g.zjob[e].t)] = lerp3((k >> (2 * JOB_BITS)) & 3, yv[k & JM], yv[(k >> JOB_BITS) & JM]);
      }
      __syncthreads();
    }
    const bool second = slot >= 0, pair = der_f32(MIXED, v);  // pair: the tile holds split pairs
    for (int t0 = threadIdx.x; t0 < T3; t0 += BATCH * THREADS) {
      double val[BATCH];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int t = t0 + u * THREADS;
        val[u] = 0.0;
        if (t >= T3) continue;
        if (SRC == FROM_TILE) {
          val[u] = __ldcs(tv + t);
        } else {
          const int s = idx[t];
          if (s >= 0) val[u] = __ldg(sv + s);
          else if (MESH && s <= -2) val[u] = __ldcg(tv + t);  // interpolated above (through L2)
        }
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int t = t0 + u * THREADS;
        if (t >= T3) continue;
        double w = val[u];
        if (SRC != FROM_TILE && tile_out) __stcs(tv + t, w);
        if (pair) {
          ts[t] = SRC == FROM_TILE ? w : split_pair(w);
        } else if (!second || SRC == FROM_TILE) {
          unsigned e;
          reinterpret_cast<int64_t *>(ts)[t] = fx_word(w, e);
          ex[t] = e;
        } else {
          ts[t] = w;
        }
      }
    }
    __syncthreads();
    if (second && SRC != FROM_TILE) {
      // the mixed derivatives, as the halo fill forms them
#pragma unroll 1
      for (int pass = 0; pass < (wide ? 1 : 3); ++pass) {
        const int si = pass == 0 ? T : T * T;
        for (int e = threadIdx.x; e < next; e += THREADS) {
          const int a = e % pe - 2, b = (e / pe) % p, c = e / (pe * p);
          const int x = pass == 2 ? b : a, y = pass == 2 ? a : b;
          mixed_in(ext, e, ts, ((c + HALO) * T + (y + HALO)) * T + (x + HALO), si, pair);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < p3; q += THREADS) {
          const int x = q % p, y = (q / p) % p, z = q / (p * p);
          const int a = pass == 2 ? y : x, b = pass == 2 ? x : y;
          mixed_out(ext, (z * p + b) * pe + (a + 2), 1, cmix, cmixf, pair, mix, np, pbase, slot + pass, q);
        }
        __syncthreads();
      }
      if (wide) {
        for (int e = threadIdx.x; e < pe * pe * p; e += THREADS) {
          const int a = e % pe - 2, b = (e / pe) % pe - 2, c = e / (pe * pe);
          if ((a < 0 || a >= p) && (b < 0 || b >= p)) continue;
          mixed_in(ext, e, ts, ((c + HALO) * T + (b + HALO)) * T + (a + HALO), T * T, pair);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < p3; q += THREADS) {
          const int x = q % p, y = (q / p) % p, z = q / (p * p);
          const int e = (z * pe + (y + 2)) * pe + (x + 2);
          mixed_out(ext, e, 1, cmix, cmixf, pair, mix, np, pbase, slot + 1, q);
          mixed_out(ext, e, pe, cmix, cmixf, pair, mix, np, pbase, slot + 2, q);
        }
      }
      if (sums && !pair) {
        __syncthreads();  // the exponents take the widened region's place
        for (int t = threadIdx.x; t < T3; t += THREADS) {
          unsigned e;
          reinterpret_cast<int64_t *>(ts)[t] = fx_word(ts[t], e);
          ex[t] = e;
        }
        __syncthreads();
      }
    }
    if (!sums) continue;
    double *dd = der + (MIXED ? (v == ALPHA ? 0 : 7) : 4 * v) * dnp + dbase;
    double *dp = MIXED ? dd + 4 * dnp : der + (4 * NF + 3 * (second ? slot / 3 : 0)) * dnp + dbase;
    float *fd = reinterpret_cast<float *>(der + DER_D * dnp) + (long long)(4 * der_f(v)) * dnp + dbase;
    float *fp = reinterpret_cast<float *>(der + DER_D * dnp) + (long long)(DER_F + 3 * der_f2(v)) * dnp + dbase;
    auto each = [&](auto is_second, auto zero) {
      using O = decltype(zero);
      constexpr bool SECOND = decltype(is_second)::value;
      auto point = [&](int q, int c0) {
        O o[7];
        if constexpr (std::is_same<O, float>::value)
          point_sums<SECOND>(reinterpret_cast<const float2 *>(ts) + c0, ex, T, o);
        // the 58 fields leave the FP64 pipe to 3 %: 25 steps at 54^3 106.4 ms with their first derivatives returned in
        // integers, 104.5 by the conversion instruction; the 25 do not (monitors 5.84 against 5.88)
        else point_sums<SECOND, true, NF != NV>(reinterpret_cast<const int64_t *>(ts) + c0, ex + c0, T, o);
        O *a, *b;
        if constexpr (std::is_same<O, float>::value) {
          a = fd + q;
          b = fp + q;
        } else {
          a = dd + q;
          b = dp + q;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) a[k * dnp] = o[k];
        if (SECOND) {
#pragma unroll
          for (int k = 0; k < 3; ++k) b[k * dnp] = o[4 + k];
        }
      };
      if (PF > 0) {
#pragma unroll 1
        for (int r = 0, q = threadIdx.x; r < ROUNDS; ++r, q += THREADS) {
          int c0 = at[0];
#pragma unroll
          for (int s = 1; s < ROUNDS; ++s) c0 = r == s ? at[s] : c0;
          if (q < p3) point(q, c0);
        }
      } else {
        for (int q = threadIdx.x; q < p3; q += THREADS) point(q, centre_at(q));
      }
    };
    if constexpr (NF != NV) {
      each(std::false_type(), 0.0);
    } else if constexpr (MIXED) {
      if (!pair) each(std::true_type(), 0.0);
      else if (second) each(std::true_type(), 0.0f);
      else each(std::false_type(), 0.0f);
    } else {
      if (second) each(std::true_type(), 0.0);
      else each(std::false_type(), 0.0);
    }
  }
}

}  // namespace

}  // namespace ccz4
