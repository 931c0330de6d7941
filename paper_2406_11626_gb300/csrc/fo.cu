// The first-order CCZ4 formulation (58 variables) and the second-order
// formulation with reconstructed auxiliary variables (Alg. fd4-fo and Alg.
// fd4-so of Sec. "Explicit gradient reconstruction"), on a single uniform
// level, FP64, behind ccz4_fo_*.
//
// A ccz4_fo holds 58-field state buffers on the geometry of a grid (its
// patches, neighbour lookup and Sommerfeld ghost shell). Per RK4 stage:
//  - first order: the derivative pass (derive.cuh) over all 58 fields, the
//    stage kernel (every variable evolved, red terms kept; ghost cells too);
//  - second order with reconstruction: the derivative pass over the 25
//    primaries, the reconstruction kernel (the auxiliary variables of every
//    interior point from the FD4 derivatives of the primaries, written into
//    the stage's input), the derivative pass over the 33 auxiliary variables,
//    the stage kernel (the primaries evolved without red terms; ghost cells
//    too); after the last stage the auxiliary variables are reconstructed
//    from the new primaries. This is the extra mesh sweep the paper's second-order
//    formulation needs.
// The ghost cells of every variable follow the radiative condition of the
// Sommerfeld boundary (speed somm_speed[v] for the primaries, 1 for the
// auxiliary variables).
#include <vector>

#include "fo_stage.cuh"

namespace ccz4 {
namespace {

// One thread per interior point: its auxiliary variables from the primaries'
// first derivatives, written into the state `out`.
__global__ void __launch_bounds__(128) fo_reconstruct_kernel(GridView g, const double *__restrict__ der,
                                                             double *__restrict__ out, double c1) {
  const long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x, p3 = g.p * g.p * g.p;
  if (q >= g.wn * p3) return;
  const long long i = g.w0 * p3 + q;
  const FoView N = fo_view(g, der, out, i, q);
  const long long S = g.S;
  auto put = [&](int v, double val) { out[v * S + i] = val; };
  fo_reconstruct_point(N, c1, put);
}

// stage -1: plain right-hand side (all 58, red terms per `red`); 0..3: RK4 stage
template <int MODE>
cudaError_t launch_fo_mode(const GridView &g, const ccz4_params &P, bool first_order, const double *der,
                           const double *in, const double *ini, const FoStageArgs &a, cudaStream_t s) {
  return first_order ? launch_fo_interior<MODE, true, true>(g, P, der, in, ini, a, s)
                     : launch_fo_interior<MODE, false, (MODE < 0)>(g, P, der, in, ini, a, s);
}

cudaError_t launch_fo(int stage, const GridView &g, const ccz4_params &P, bool first_order, const double *der,
                      const double *in, const double *ini, const FoStageArgs &a, cudaStream_t s) {
  switch (stage) {
    case -1: return launch_fo_mode<-1>(g, P, first_order, der, in, ini, a, s);
    case 0: return launch_fo_mode<0>(g, P, first_order, der, in, ini, a, s);
    case 1: return launch_fo_mode<1>(g, P, first_order, der, in, ini, a, s);
    case 2: return launch_fo_mode<2>(g, P, first_order, der, in, ini, a, s);
    case 3: return launch_fo_mode<3>(g, P, first_order, der, in, ini, a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace
}  // namespace ccz4

using namespace ccz4;

struct ccz4_fo {
  ccz4_grid *g;
  int variant;
  double *buf[6];  // U, Y0, Y1, ACC, RHS, INI: [58][S]
  GridView v;      // the grid's, with the windows of this derivative buffer
  double *der;     // derivative buffer, [4 x 58][v.wcap p^3]
};

static const int kFoIn[4] = {CCZ4_BUF_U, CCZ4_BUF_Y0, CCZ4_BUF_Y1, CCZ4_BUF_Y0};
static const int kFoOut[4] = {CCZ4_BUF_Y0, CCZ4_BUF_Y1, CCZ4_BUF_Y0, CCZ4_BUF_U};

#define FO_TRY(call)                                                               \
  do {                                                                             \
    cudaError_t e_ = (call);                                                       \
    if (e_ != cudaSuccess) {                                                       \
      set_error("%s failed: %s", #call, cudaGetErrorString(e_));                   \
      return CCZ4_ERR_CUDA;                                                        \
    }                                                                              \
  } while (0)

static void fo_release(ccz4_fo *f) {
  if (!f) return;
  for (double *b : f->buf) cudaFree(b);
  cudaFree(f->der);
  free(f);
}

// f on the view of each window of the formulation's derivative buffer.
template <class F>
static cudaError_t fo_windows(const ccz4_fo *f, F call) {
  GridView w = f->v;
  cudaError_t e = cudaSuccess;
  for (w.w0 = 0; w.w0 < w.n_patches && e == cudaSuccess; w.w0 += w.wcap) {
    w.wn = w.n_patches - w.w0 < w.wcap ? w.n_patches - w.w0 : w.wcap;
    e = call(w);
  }
  return e;
}

// The derivative pass over fields [v0, v0 + nv) of a window.
static cudaError_t fo_derive(const ccz4_fo *f, const GridView &w, const double *src, int v0, int nv, cudaStream_t s) {
  FieldList fl;
  fl.n = nv;
  for (int k = 0; k < nv; ++k) fl.f[k] = (unsigned char)(v0 + k);
  return launch_derive_fo(w, src, f->der, fl, s);
}

static cudaError_t fo_reconstruct_into(const ccz4_fo *f, double *state, cudaStream_t s) {
  return fo_windows(f, [&](const GridView &w) {
    const cudaError_t e = fo_derive(f, w, state, 0, NV, s);
    if (e != cudaSuccess) return e;
    const long long points = (long long)w.wn * w.p * w.p * w.p;
    fo_reconstruct_kernel<<<(unsigned)((points + 127) / 128), 128, 0, s>>>(w, f->der, state, 1.0 / (12.0 * w.dx));
    return cudaGetLastError();
  });
}

// The right-hand side or a stage (launch_fo) of every window, from the derivatives of fields [v0, 58) and
// those that the buffer holds already.
static cudaError_t fo_stage_windows(const ccz4_fo *f, int stage, const ccz4_params &P, bool first, const double *in,
                                    int v0, const double *ini, const FoStageArgs &a, cudaStream_t s) {
  return fo_windows(f, [&](const GridView &w) {
    const cudaError_t e = fo_derive(f, w, in, v0, NVF - v0, s);
    return e == cudaSuccess ? launch_fo(stage, w, P, first, f->der, in, ini, a, s) : e;
  });
}

static const double *fo_ini(const ccz4_fo *f) {
  return f->buf[CCZ4_BUF_INI] ? f->buf[CCZ4_BUF_INI] : f->buf[CCZ4_BUF_U];
}

static bool fo_check(const ccz4_fo *f, const ccz4_params *P) {
  if (!f || !P) {
    set_error("fo: handle and parameters must be given");
    return false;
  }
  return true;
}

extern "C" ccz4_status ccz4_fo_alloc(ccz4_grid *g, int variant, ccz4_fo **out) {
  if (!out || !g) {
    set_error("fo_alloc: grid and out must be given");
    return CCZ4_ERR_INVALID;
  }
  *out = nullptr;
  if (variant != CCZ4_FO_FIRST_ORDER && variant != CCZ4_FO_SO_RECONSTRUCT) {
    set_error("fo_alloc: unknown variant %d", variant);
    return CCZ4_ERR_INVALID;
  }
  if (g->v.n_levels > 1 || g->v.src) {
    set_error("fo_alloc: the 58-variable formulations run on a single uniform level, not on a refined mesh");
    return CCZ4_ERR_INVALID;
  }
  ccz4_fo *f = (ccz4_fo *)calloc(1, sizeof(ccz4_fo));
  if (!f) {
    set_error("host allocation failed");
    return CCZ4_ERR_NOMEM;
  }
  f->g = g;
  f->variant = variant;
  const GridView &v = g->v;
  const size_t state = sizeof(double) * (size_t)NVF * (size_t)v.S;
  for (int b = 0; b < 6; ++b) {
    if (b == CCZ4_BUF_INI && v.n_ghost == 0) continue;
    if (cudaMalloc(&f->buf[b], state) != cudaSuccess || cudaMemset(f->buf[b], 0, state) != cudaSuccess) {
      set_error("fo_alloc: cudaMalloc of %zu bytes failed: %s", state, cudaGetErrorString(cudaGetLastError()));
      fo_release(f);
      return CCZ4_ERR_NOMEM;
    }
  }
  f->v = v;
  for (f->v.wcap = fitting_window(v, 4 * NVF); v.n_points > 0;) {
    const size_t der = sizeof(double) * 4 * (size_t)NVF * (size_t)f->v.wcap * (size_t)(v.p * v.p * v.p);
    if (cudaMalloc(&f->der, der) == cudaSuccess) break;
    f->der = nullptr;
    const cudaError_t e = cudaGetLastError();
    f->v.wcap = smaller_window(v, f->v.wcap);
    if (f->v.wcap > 0) continue;
    set_error("fo_alloc: cudaMalloc of the %zu-byte derivative buffer failed: %s", der, cudaGetErrorString(e));
    fo_release(f);
    return CCZ4_ERR_NOMEM;
  }
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) {
    set_error("fo_alloc: set-up failed: %s", cudaGetErrorString(e));
    fo_release(f);
    return CCZ4_ERR_CUDA;
  }
  *out = f;
  return CCZ4_OK;
}

extern "C" ccz4_status ccz4_fo_free(ccz4_fo *f) {
  fo_release(f);
  return CCZ4_OK;
}

static ccz4_status fo_copy(ccz4_fo *f, int buf, double *U, double *G, bool to_device, cudaStream_t s) {
  if (!f || buf < CCZ4_BUF_U || buf > CCZ4_BUF_INI || !f->buf[buf] || !U) {
    set_error("fo upload/download: handle, a state buffer of this formulation (U..INI) and U must be given");
    return CCZ4_ERR_INVALID;
  }
  const GridView &v = f->g->v;
  if (v.n_ghost > 0 && !G) {
    set_error("fo upload/download: this grid has %lld Sommerfeld ghost cells; G must be given", v.n_ghost);
    return CCZ4_ERR_INVALID;
  }
  const size_t dp = sizeof(double) * (size_t)v.S;
  double *d = f->buf[buf];
  if (to_device) {
    FO_TRY(cudaMemcpy2DAsync(d, dp, U, sizeof(double) * v.n_points, sizeof(double) * v.n_points, NVF,
                             cudaMemcpyHostToDevice, s));
    if (v.n_ghost)
      FO_TRY(cudaMemcpy2DAsync(d + v.n_points, dp, G, sizeof(double) * v.n_ghost, sizeof(double) * v.n_ghost, NVF,
                               cudaMemcpyHostToDevice, s));
  } else {
    back_host_pages(U, sizeof(double) * (size_t)v.n_points * NVF);
    if (v.n_ghost) back_host_pages(G, sizeof(double) * (size_t)v.n_ghost * NVF);
    FO_TRY(cudaMemcpy2DAsync(U, sizeof(double) * v.n_points, d, dp, sizeof(double) * v.n_points, NVF,
                             cudaMemcpyDeviceToHost, s));
    if (v.n_ghost)
      FO_TRY(cudaMemcpy2DAsync(G, sizeof(double) * v.n_ghost, d + v.n_points, dp, sizeof(double) * v.n_ghost, NVF,
                               cudaMemcpyDeviceToHost, s));
  }
  FO_TRY(cudaStreamSynchronize(s));
  return CCZ4_OK;
}

extern "C" ccz4_status ccz4_fo_upload(ccz4_fo *f, int buf, const double *U, const double *G, void *stream) {
  return fo_copy(f, buf, const_cast<double *>(U), const_cast<double *>(G), true, (cudaStream_t)stream);
}

extern "C" ccz4_status ccz4_fo_download(ccz4_fo *f, int buf, double *U, double *G, void *stream) {
  return fo_copy(f, buf, U, G, false, (cudaStream_t)stream);
}

extern "C" ccz4_status ccz4_fo_reconstruct(ccz4_fo *f, int buf, void *stream) {
  if (!f || buf < CCZ4_BUF_U || buf > CCZ4_BUF_INI || !f->buf[buf]) {
    set_error("fo_reconstruct: handle and a state buffer (U..INI) must be given");
    return CCZ4_ERR_INVALID;
  }
  FO_TRY(fo_reconstruct_into(f, f->buf[buf], (cudaStream_t)stream));
  return CCZ4_OK;
}

extern "C" ccz4_status ccz4_fo_rhs(ccz4_fo *f, const ccz4_params *P, int in_buf, int out_buf, void *stream) {
  if (!fo_check(f, P)) return CCZ4_ERR_INVALID;
  if (in_buf < CCZ4_BUF_U || in_buf > CCZ4_BUF_INI || out_buf < CCZ4_BUF_U || out_buf > CCZ4_BUF_INI ||
      in_buf == out_buf || !f->buf[in_buf] || !f->buf[out_buf]) {
    set_error("fo_rhs: in and out must be distinct state buffers of this formulation");
    return CCZ4_ERR_INVALID;
  }
  cudaStream_t s = (cudaStream_t)stream;
  const double *in = f->buf[in_buf];
  FoStageArgs a{nullptr, nullptr, f->buf[out_buf], 0.0};
  FO_TRY(fo_stage_windows(f, -1, *P, f->variant == CCZ4_FO_FIRST_ORDER, in, 0, fo_ini(f), a, s));
  return CCZ4_OK;
}

// One RK4 stage: the derivatives (and, second order, the reconstruction) and
// the stage kernel; stage 3 ends the step (enforcement in
// the stage kernel; second order: the auxiliary variables of U_{n+1}
// reconstructed).
static ccz4_status fo_stage(ccz4_fo *f, const ccz4_params *P, int stage, double dt, cudaStream_t s) {
  double *in = f->buf[kFoIn[stage]];
  const bool first = f->variant == CCZ4_FO_FIRST_ORDER;
  if (!first) FO_TRY(fo_reconstruct_into(f, in, s));
  // (one window: the reconstruction has left the primaries' derivatives in the buffer)
  const int v0 = !first && f->v.wcap >= f->v.n_patches ? NV : 0;
  FoStageArgs a{f->buf[CCZ4_BUF_U], f->buf[CCZ4_BUF_ACC], f->buf[kFoOut[stage]], dt};
  FO_TRY(fo_stage_windows(f, stage, *P, first, in, v0, fo_ini(f), a, s));
  if (stage == 3 && !first) FO_TRY(fo_reconstruct_into(f, f->buf[CCZ4_BUF_U], s));
  return CCZ4_OK;
}

extern "C" ccz4_status ccz4_fo_rk_stage(ccz4_fo *f, const ccz4_params *P, int stage, double dt, void *stream) {
  if (!fo_check(f, P)) return CCZ4_ERR_INVALID;
  if (stage < 0 || stage > 3 || !(dt == dt)) {
    set_error("fo_rk_stage: stage must be 0..3 (got %d) and dt finite", stage);
    return CCZ4_ERR_INVALID;
  }
  return fo_stage(f, P, stage, dt, (cudaStream_t)stream);
}

extern "C" ccz4_status ccz4_fo_step(ccz4_fo *f, const ccz4_params *P, double dt, int n_steps, void *stream) {
  if (!fo_check(f, P)) return CCZ4_ERR_INVALID;
  if (n_steps < 0 || !(dt == dt)) {
    set_error("fo_step: n_steps must be >= 0 and dt finite");
    return CCZ4_ERR_INVALID;
  }
  for (int n = 0; n < n_steps; ++n)
    for (int st = 0; st < 4; ++st) {
      ccz4_status r = fo_stage(f, P, st, dt, (cudaStream_t)stream);
      if (r != CCZ4_OK) return r;
    }
  return CCZ4_OK;
}
