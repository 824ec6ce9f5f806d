// wos_render.cu -- headless view of a progressive solve on a slice plane (Sec. 7.2:
// signed-distance geometry rendered by sphere tracing, the solution shown on a slice
// plane and refined by accumulating one walk per point per frame).
//
// wos_slice_points lays the slice grid out (cell centres of an nu x nv grid on the
// plane rectangle); the walks run through the ordinary solve entry points and add to
// per-point accumulators; wos_render_slice then draws, per pixel, a pinhole ray that
// is sphere-traced against the domain clipped by the slice plane (the part of the
// domain on the camera's side of the plane is cut away).  A ray that reaches the
// plane inside the domain shows the accumulated mean of its slice cell through a
// colour map; a ray that reaches the boundary shows g there, shaded by the surface
// normal.  2D problems show the slice grid directly (the plane is the domain's own
// plane).  The output is an RGBA8 image in device memory, plus optional per-pixel
// value (NaN off the slice) and ray depth (INFINITY on a miss) buffers.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <cmath>

#include "wos.h"
#include "wos_math.cuh"
#include "wos_problem.cuh"

namespace wos {
namespace {

struct View3 {
  double eye[3], fwd[3], right[3], up[3];
  double tan_half;
  double org[3], pu[3], pv[3], n[3];  // plane rectangle and its normal (towards the eye)
  double pu2, pv2;
  double lo, hi;
  double scale;                        // size of the domain box, for tolerances
  int nu, nv, width, height;
};

__device__ double sd_domain(const DevProblem<double>& P, const double* x) {
  double xb[3];
  return -distance<3, double, false>(P, x, xb);  // signed distance, negative inside
}

// A CSG list in FP32, with a bound of the FP32 distances' error: the sphere tracer asks it which
// primitive decides the signed distance, and evaluates that one alone in FP64.
//
// What bounds the view is the FP64 pipe (1/64 of the FP32 lanes' rate here): every step of a ray
// evaluated the plane and every primitive in FP64, some 25 operations each with a square root.  The
// FP32 pass costs a fraction of that; where its intervals do not tell the winner (a crease, a far-off
// point) the whole list is evaluated in FP64 as before, so every step's length, and the image, is
// the same.  Measured (1280 x 720, five primitives): 5.70 -> 2.33 ms, FP64 instructions 74 % of their peak; more
// resident blocks by spilling (3, 4 or 5 of 256 threads) 2.8, 2.9 and 4.3 ms.
struct CsgF32 {
  CsgNode<float> node[kMaxCsg];
  float size[kMaxCsg];   // largest parameter, times (1 + its normal's) for a half-space
};

__device__ void csg_load_f32(const DevProblem<double>& P, CsgF32* C) {
  for (int i = threadIdx.x; i < P.ncsg; i += blockDim.x) {
    C->node[i].prim = P.csg[i].prim;
    C->node[i].op = P.csg[i].op;
    float m = 0.0f;
    for (int k = 0; k < 8; ++k) {
      C->node[i].p[k] = (float)P.csg[i].p[k];
      m = fmaxf(m, fabsf(C->node[i].p[k]));
    }
    C->size[i] = m * (P.csg[i].prim == C_HALFSPACE ? 1.0f + m : 1.0f);
  }
}

// The interval [lo, hi] of csg_sdf at a point and the primitive that gives it, -1 where that is open
// (an unbounded interval if some distance is not finite).  xf is the point in FP32, off by a few
// roundings of numbers no larger than X (>= the sum of its coordinates' magnitudes).  A primitive's
// FP32 distance takes at most a few dozen roundings of numbers no larger than X plus its parameters
// (a half-space: times its normal's length): 64 units of 2^-24 bound its error.
__device__ int csg_decide(const CsgF32& C, int n, const float* xf, float X, float* lo, float* hi) {
  float l = 0.0f, h = 0.0f;
  int who = 0;
  bool finite = true;
  for (int i = 0; i < n; ++i) {
    float g[3];
    const int op = C.node[i].op;
    float s = csg_prim<3, float>(C.node[i], xf, g);
    const float grow = C.node[i].prim == C_HALFSPACE ? 1.0f + C.size[i] : 1.0f;
    const float e = 64.0f * 5.9604645e-8f * (X * grow + C.size[i]);
    if (i > 0 && op == C_SUBTRACT) s = -s;
    const float a = s - e, b = s + e;
    finite = finite && fabsf(a) < INFINITY && fabsf(b) < INFINITY;
    if (i == 0) {
      l = a;
      h = b;
    } else if (op == C_UNION) {   // the smaller
      if (b < l) {
        who = i;
        l = a;
        h = b;
      } else if (!(a > h)) {
        who = -1;
        l = fminf(l, a);
        h = fminf(h, b);
      }
    } else {                      // the larger
      if (a > h) {
        who = i;
        l = a;
        h = b;
      } else if (!(b < l)) {
        who = -1;
        l = fmaxf(l, a);
        h = fmaxf(h, b);
      }
    }
  }
  *lo = finite ? l : -INFINITY;
  *hi = finite ? h : INFINITY;
  return finite ? who : -1;
}

// sd_domain of a CSG list through csg_decide
__device__ double sd_decided(const DevProblem<double>& P, const CsgF32& C, const double* x) {
  const float xf[3] = {(float)x[0], (float)x[1], (float)x[2]};
  float lo, hi;
  const int who = csg_decide(C, P.ncsg, xf, fabsf(xf[0]) + fabsf(xf[1]) + fabsf(xf[2]), &lo, &hi);
  if (who < 0) return sd_domain(P, x);
  double g[3];
  const double s = csg_prim<3, double>(P.csg[who], x, g);
  return (who > 0 && P.csg[who].op == C_SUBTRACT) ? -s : s;
}

__device__ void colour_map(double t, double* c) {
  // a blue - white - red map on [0, 1]
  t = fmin(fmax(t, 0.0), 1.0);
  if (t < 0.5) {
    double s = t * 2.0;
    c[0] = 0.23 + 0.77 * s; c[1] = 0.30 + 0.70 * s; c[2] = 0.75 + 0.25 * s;
  } else {
    double s = (t - 0.5) * 2.0;
    c[0] = 1.0 - 0.29 * s; c[1] = 1.0 - 0.98 * s; c[2] = 1.0 - 0.85 * s;
  }
}

__device__ void put(uint8_t* rgba, int64_t i, const double* c) {
  for (int k = 0; k < 3; ++k) rgba[4 * i + k] = (uint8_t)fmin(255.0, fmax(0.0, c[k] * 255.0 + 0.5));
  rgba[4 * i + 3] = 255;
}

// CSG: the domain is a CSG list, and csg_decide chooses what a step evaluates.  A form of its own, since its
// registers (86 a thread against 78) slowed the views of other domains down (a box 972 -> 1,018 us).
template <bool CSG>
__global__ void render3_kernel(const DevProblem<double>* Pg, View3 V, const double* sum, const int64_t* count,
                               uint8_t* rgba, float* value, float* depth) {
  const DevProblem<double>& P = *Pg;
  __shared__ CsgF32 C;
  if (CSG) {
    csg_load_f32(P, &C);
    __syncthreads();
  }
  int64_t npx = (int64_t)V.width * V.height;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx; i += (int64_t)gridDim.x * blockDim.x) {
    int px = (int)(i % V.width), py = (int)(i / V.width);
    double sx = ((px + 0.5) / V.width * 2.0 - 1.0) * V.tan_half * V.width / V.height;
    double sy = (1.0 - (py + 0.5) / V.height * 2.0) * V.tan_half;
    double dir[3], nd = 0.0;
    for (int k = 0; k < 3; ++k) {
      dir[k] = V.fwd[k] + sx * V.right[k] + sy * V.up[k];
      nd += dir[k] * dir[k];
    }
    nd = sqrt(nd);
    for (int k = 0; k < 3; ++k) dir[k] /= nd;
    double c[3] = {0.08, 0.08, 0.10};
    float val = NAN, dep = INFINITY;
    // sphere-trace max(sdf_domain, sdf_keep): the domain behind the plane
    double t = 0.0, tmax = 1e3 * V.scale;
    float eyef[3], dirf[3], nf[3], orgf[3], eye1 = 0.0f, org1 = 0.0f;
    for (int k = 0; CSG && k < 3; ++k) {
      eyef[k] = (float)V.eye[k];
      dirf[k] = (float)dir[k];
      nf[k] = (float)V.n[k];
      orgf[k] = (float)V.org[k];
      eye1 += fabsf(eyef[k]);
      org1 += fabsf(orgf[k]);
    }
    const double tol = 1e-5 * V.scale;
    for (int it = 0; it < 512 && t < tmax; ++it) {
      double x[3];
      for (int k = 0; k < 3; ++k) x[k] = V.eye[k] + t * dir[k];
      // which of the domain's and the plane's distance is the larger, in FP32 where that suffices
      bool plane = true, domain = true;  // may be
      int who = -1;
      if (CSG) {
        const float tf = (float)t, X = eye1 + 1.75f * fabsf(tf);
        float xf[3], spf = 0.0f, lo, hi;
        for (int k = 0; k < 3; ++k) {
          xf[k] = eyef[k] + tf * dirf[k];
          spf += nf[k] * (xf[k] - orgf[k]);
        }
        who = csg_decide(C, P.ncsg, xf, X, &lo, &hi);
        const float e = 64.0f * 5.9604645e-8f * (X + org1);
        plane = !(spf + e < lo);
        domain = !(hi < spf - e);
      }
      double sd = -INFINITY, sp = -INFINITY;
      if (plane) {  // > 0 on the eye's side of the plane: cut away
        sp = 0.0;
        for (int k = 0; k < 3; ++k) sp += V.n[k] * (x[k] - V.org[k]);
      }
      if (domain) {
        if (who >= 0) {
          double g[3];
          sd = csg_prim<3, double>(P.csg[who], x, g);
          if (who > 0 && P.csg[who].op == C_SUBTRACT) sd = -sd;
        } else {
          sd = sd_domain(P, x);
        }
      }
      double s = fmax(sd, sp);
      if (s < tol) {
        dep = (float)t;
        if (sp >= sd) {
          // on the slice plane, inside the domain
          double r[3], a = 0.0, b = 0.0;
          for (int k = 0; k < 3; ++k) r[k] = x[k] - V.org[k];
          for (int k = 0; k < 3; ++k) { a += r[k] * V.pu[k]; b += r[k] * V.pv[k]; }
          a /= V.pu2;
          b /= V.pv2;
          if (a >= 0.0 && a < 1.0 && b >= 0.0 && b < 1.0) {
            int iu = min((int)(a * V.nu), V.nu - 1), iv = min((int)(b * V.nv), V.nv - 1);
            int64_t cell = (int64_t)iv * V.nu + iu;
            int64_t n = count[cell];
            if (n > 0) {
              double u = sum[cell] / (double)n;
              val = (float)u;
              colour_map((u - V.lo) / (V.hi - V.lo), c);
            } else {
              c[0] = c[1] = c[2] = 0.35;
            }
          } else {
            c[0] = c[1] = c[2] = 0.25;
          }
        } else {
          // boundary: g there, Lambert-shaded by the normal of the signed distance
          double h = 1e-4 * V.scale, g[3];
          for (int k = 0; k < 3; ++k) {
            double xp[3] = {x[0], x[1], x[2]}, xm[3] = {x[0], x[1], x[2]};
            xp[k] += h;
            xm[k] -= h;
            g[k] = CSG ? sd_decided(P, C, xp) - sd_decided(P, C, xm) : sd_domain(P, xp) - sd_domain(P, xm);
          }
          double gn = sqrt(g[0] * g[0] + g[1] * g[1] + g[2] * g[2]) + 1e-300;
          double lam = 0.0;
          for (int k = 0; k < 3; ++k) lam -= g[k] / gn * dir[k];
          lam = 0.25 + 0.75 * fmax(lam, 0.0);
          double gv = field_eval<3>(P, P.g, x[0], x[1], x[2], false).v;
          colour_map((gv - V.lo) / (V.hi - V.lo), c);
          for (int k = 0; k < 3; ++k) c[k] *= lam;
        }
        break;
      }
      t += fmax(s, tol);
    }
    put(rgba, i, c);
    if (value) value[i] = val;
    if (depth) depth[i] = dep;
  }
}

__global__ void render2_kernel(const DevProblem<double>* Pg, double o0, double o1, double u0, double v1, int nu,
                               int nv, int width, int height, double lo, double hi, const double* sum,
                               const int64_t* count, uint8_t* rgba, float* value) {
  const DevProblem<double>& P = *Pg;
  int64_t npx = (int64_t)width * height;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx; i += (int64_t)gridDim.x * blockDim.x) {
    int px = (int)(i % width), py = (int)(i / width);
    double a = (px + 0.5) / width, b = 1.0 - (py + 0.5) / height;
    double x[3] = {o0 + a * u0, o1 + b * v1, 0.0}, xb[3];
    double c[3] = {0.08, 0.08, 0.10};
    float val = NAN;
    if (distance<2, double, false>(P, x, xb) > 0.0) {
      int iu = min((int)(a * nu), nu - 1), iv = min((int)(b * nv), nv - 1);
      int64_t cell = (int64_t)iv * nu + iu;
      int64_t n = count[cell];
      if (n > 0) {
        double u = sum[cell] / (double)n;
        val = (float)u;
        colour_map((u - lo) / (hi - lo), c);
      } else {
        c[0] = c[1] = c[2] = 0.35;
      }
    }
    put(rgba, i, c);
    if (value) value[i] = val;
  }
}

__global__ void slice_points_kernel(int dim, View3 V, float* pts) {
  int64_t n = (int64_t)V.nu * V.nv;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double a = ((i % V.nu) + 0.5) / V.nu, b = ((i / V.nu) + 0.5) / V.nv;
    for (int k = 0; k < dim; ++k) pts[(int64_t)k * n + i] = (float)(V.org[k] + a * V.pu[k] + b * V.pv[k]);
  }
}

double dot3(const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }
void cross3(const double* a, const double* b, double* c) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}
bool normalise(double* a) {
  double n = sqrt(dot3(a, a));
  if (!(n > 0.0) || !std::isfinite(n)) return false;
  for (int k = 0; k < 3; ++k) a[k] /= n;
  return true;
}

bool make_view(const wos_view* v, int dim, View3* V) {
  for (int k = 0; k < 3; ++k) {
    V->org[k] = v->plane_origin[k];
    V->pu[k] = v->plane_u[k];
    V->pv[k] = v->plane_v[k];
  }
  if (dim == 2) {
    V->pu[1] = V->pu[2] = 0.0;
    V->pv[0] = V->pv[2] = 0.0;
    V->org[2] = 0.0;
  }
  V->pu2 = dot3(V->pu, V->pu);
  V->pv2 = dot3(V->pv, V->pv);
  V->nu = v->slice_nu;
  V->nv = v->slice_nv;
  V->width = v->width;
  V->height = v->height;
  V->lo = v->value_lo;
  V->hi = v->value_hi;
  if (!(V->pu2 > 0.0) || !(V->pv2 > 0.0) || V->nu < 1 || V->nv < 1) return false;
  if (dim == 2) return true;
  cross3(V->pu, V->pv, V->n);
  if (!normalise(V->n)) return false;
  for (int k = 0; k < 3; ++k) {
    V->eye[k] = v->eye[k];
    V->fwd[k] = v->look[k] - v->eye[k];
  }
  if (!normalise(V->fwd)) return false;
  double up[3] = {v->up[0], v->up[1], v->up[2]};
  cross3(V->fwd, up, V->right);
  if (!normalise(V->right)) return false;
  cross3(V->right, V->fwd, V->up);
  V->tan_half = tan(0.5 * v->fov_y_deg * 3.14159265358979323846 / 180.0);
  if (!(V->tan_half > 0.0) || !std::isfinite(V->tan_half)) return false;
  // the plane normal points to the eye's side (that half is cut away)
  double r[3];
  for (int k = 0; k < 3; ++k) r[k] = V->eye[k] - V->org[k];
  if (dot3(r, V->n) < 0.0)
    for (int k = 0; k < 3; ++k) V->n[k] = -V->n[k];
  return true;
}

}  // namespace

int render_slice(const DevProblem<double>* dprob, const DevProblem<double>& host, int dim, const wos_view* view,
                 const double* sum, const int64_t* count, uint8_t* rgba, float* value, float* depth, int num_sms,
                 cudaStream_t st) {
  View3 V;
  if (!make_view(view, dim, &V)) return WOS_EINVAL;
  if (V.width < 1 || V.height < 1 || !(V.hi > V.lo)) return WOS_EINVAL;
  int64_t npx = (int64_t)V.width * V.height;
  int blocks = (int)((npx + 255) / 256);
  if (blocks > num_sms * 16) blocks = num_sms * 16;
  if (dim == 2) {
    render2_kernel<<<blocks, 256, 0, st>>>(dprob, V.org[0], V.org[1], V.pu[0], V.pv[1], V.nu, V.nv, V.width,
                                           V.height, V.lo, V.hi, sum, count, rgba, value);
  } else {
    double span2 = 0.0;
    for (int k = 0; k < 3; ++k) span2 += (host.dom[3 + k] - host.dom[k]) * (host.dom[3 + k] - host.dom[k]);
    V.scale = sqrt(span2) > 0.0 ? sqrt(span2) : 1.0;
    auto* kernel = host.domain_kind == D_CSG ? render3_kernel<true> : render3_kernel<false>;
    kernel<<<blocks, 256, 0, st>>>(dprob, V, sum, count, rgba, value, depth);
  }
  return cudaGetLastError() == cudaSuccess ? WOS_OK : WOS_ECUDA;
}

int slice_points(int dim, const wos_view* view, float* pts, int num_sms, cudaStream_t st) {
  View3 V;
  if (!make_view(view, dim, &V)) return WOS_EINVAL;
  int64_t n = (int64_t)V.nu * V.nv;
  int blocks = (int)((n + 255) / 256);
  if (blocks > num_sms * 16) blocks = num_sms * 16;
  slice_points_kernel<<<blocks, 256, 0, st>>>(dim, V, pts);
  return cudaGetLastError() == cudaSuccess ? WOS_OK : WOS_ECUDA;
}

}  // namespace wos
