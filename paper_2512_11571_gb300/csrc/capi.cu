// C ABI of the cemtamp library: argument validation, the per-handle device
// scene and workspaces, and the device-resident CE loop of Algorithm 1
// (Sec. III-B) with one iteration captured in a CUDA graph.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <map>
#include <sstream>
#include <string>
#include <vector>

#include "internal.h"
#include "plan.cuh"

using namespace cem;

namespace {
thread_local std::string g_err;

int fail(int code, const std::string& msg) {
  g_err = msg;
  return code;
}

int cuda_fail(cudaError_t e, const char* where) {
  return fail(e == cudaErrorMemoryAllocation ? CEM_ERR_NO_MEMORY : CEM_ERR_CUDA,
              std::string(where) + ": " + cudaGetErrorString(e));
}

// the test hook's countdown: 0 = off, k = the k-th next device allocation fails
std::atomic<int> g_fail_alloc{0};

#define CEM_CUDA(call)                               \
  do {                                               \
    cudaError_t e_ = (call);                         \
    if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
  } while (0)

bool is_device_ptr(const void* p) {
  if (!p) return false;
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

// Mean distance from the centre of a 2a x 2b rectangle, closed form of
// (1/ab) * integral over [0,a]x[0,b] of sqrt(x^2 + y^2).
double mean_radius(double a, double b) {
  const double d = std::sqrt(a * a + b * b);
  const double s = a * b * d / 3.0 + a * a * a / 6.0 * std::log((b + d) / a) + b * b * b / 6.0 * std::log((a + d) / b);
  return s / (a * b);
}

int action_width(int kind) { return kind == CEM_ACT_GRASP ? 2 : 3; }
}  // namespace

struct cem_ctx {
  cem_scene_desc desc;
  cem_skeleton_desc skel;
  DevScene host;
  DevScene* scene_d = nullptr;
  int block = 0;  // rollout threads per block (0 = heuristic)
  int tpr = 1;    // lanes per pick-and-place rollout (1, 8 or 32)
  bool dr_on = false;  // domain randomisation (cem_set_randomization)
  DrArgs dr{};         // its settings; iteration and problem are filled per launch
  // workspaces of cem_solve
  int cap_N = 0, cap_K = 0, cap_iters = 0;
  float* theta_d = nullptr;
  float* J_d = nullptr;
  uint8_t* cls_d = nullptr;
  float* mean_d = nullptr;
  float* cov_d = nullptr;
  float* chol_d = nullptr;
  int32_t* keff_d = nullptr;
  int32_t* status_d = nullptr;
  Track* track_d = nullptr;
  float* hist_J_d = nullptr;
  int32_t* hist_keff_d = nullptr;
  int32_t* hist_cnt_d = nullptr;
  // the small solve state (track, status, k_eff, mean, cov, chol, histories)
  // lives in one device block carved into the pointers above, mirrored by a
  // pinned host block: a solve moves it in one copy each way
  unsigned char* state_d = nullptr;
  unsigned char* state_h = nullptr;
  cudaStream_t stream = nullptr;
  cudaGraphExec_t graph = nullptr;
  int graph_N = -1, graph_K = -1, graph_cov = -1;
  uint64_t graph_seed = 0;
  uint32_t graph_problem = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

namespace {

// ---- base planner graph (A* moveTo controller), built once per scene in FP64
// Footprint of body g: its slabs with a horizontal normal, every finite
// bound moved out by r.
struct HostFootprint {
  int n;
  double nx[CEM_MAX_SLABS], ny[CEM_MAX_SLABS], lo[CEM_MAX_SLABS], hi[CEM_MAX_SLABS];
};

bool host_footprint(const cem_geom& g, double r, HostFootprint& f) {
  f.n = 0;
  for (int i = 0; i < g.n_slabs; ++i) {
    const cem_slab& sl = g.slab[i];
    if (sl.n[2] != 0.0f) continue;
    const double lo = sl.lo, hi = sl.hi;
    f.nx[f.n] = sl.n[0];
    f.ny[f.n] = sl.n[1];
    f.lo[f.n] = std::fabs(lo) < 1e6 ? lo - r : lo;
    f.hi[f.n] = std::fabs(hi) < 1e6 ? hi + r : hi;
    ++f.n;
  }
  return f.n > 0;
}

bool host_inside(const HostFootprint& f, double x, double y) {
  for (int i = 0; i < f.n; ++i) {
    const double p = f.nx[i] * x + f.ny[i] * y;
    if (!(p > f.lo[i] && p < f.hi[i])) return false;
  }
  return true;
}

// does the open segment a -> b cross the footprint's interior (clipping the
// segment parameter against every slab)?
bool host_crosses(const HostFootprint& f, double ax, double ay, double bx, double by) {
  double t0 = 0.0, t1 = 1.0;
  for (int i = 0; i < f.n; ++i) {
    const double p0 = f.nx[i] * ax + f.ny[i] * ay, dp = f.nx[i] * (bx - ax) + f.ny[i] * (by - ay);
    const double lo = f.lo[i] + 1e-9, hi = f.hi[i] - 1e-9;
    if (std::fabs(dp) < 1e-15) {
      if (p0 <= lo || p0 >= hi) return false;
      continue;
    }
    const double ta = (lo - p0) / dp, tb = (hi - p0) / dp;
    t0 = std::max(t0, std::min(ta, tb));
    t1 = std::min(t1, std::max(ta, tb));
    if (t0 >= t1) return false;
  }
  return t0 < t1;
}

// corners of the grown footprints (pushed 1 mm out, outside every grown
// footprint) and their mutual visibility; -1 if there are more than
// CEM_MAX_CORNERS
int build_base_graph(const cem_scene_desc& s, DevScene& d) {
  HostFootprint fp[CEM_MAX_GEOMS];
  int nf = 0;
  for (int g = 0; g < s.n_geoms; ++g)
    if (s.geom[g].collide_base && host_footprint(s.geom[g], s.base_inflate, fp[nf])) ++nf;
  std::vector<double> cx, cy;
  for (int k = 0; k < nf; ++k) {
    const HostFootprint& f = fp[k];
    for (int i = 0; i < f.n; ++i)
      for (int j = i + 1; j < f.n; ++j)
        for (int ui = 0; ui < 2; ++ui)
          for (int uj = 0; uj < 2; ++uj) {
            const double bi = ui ? f.hi[i] : f.lo[i], bj = uj ? f.hi[j] : f.lo[j];
            if (std::fabs(bi) >= 1e6 || std::fabs(bj) >= 1e6) continue;
            const double det = f.nx[i] * f.ny[j] - f.ny[i] * f.nx[j];
            if (std::fabs(det) < 1e-12) continue;
            double x = (bi * f.ny[j] - bj * f.ny[i]) / det, y = (f.nx[i] * bj - f.nx[j] * bi) / det;
            bool on = true;
            for (int m = 0; m < f.n && on; ++m)
              if (m != i && m != j) {
                const double p = f.nx[m] * x + f.ny[m] * y;
                on = p >= f.lo[m] - 1e-9 && p <= f.hi[m] + 1e-9;
              }
            if (!on) continue;
            const double ox = (ui ? f.nx[i] : -f.nx[i]) + (uj ? f.nx[j] : -f.nx[j]);
            const double oy = (ui ? f.ny[i] : -f.ny[i]) + (uj ? f.ny[j] : -f.ny[j]);
            const double len = std::sqrt(ox * ox + oy * oy);
            x += 1e-3 * ox / len;
            y += 1e-3 * oy / len;
            bool clear = true;
            for (int q = 0; q < nf && clear; ++q) clear = !host_inside(fp[q], x, y);
            if (!clear) continue;
            cx.push_back(x);
            cy.push_back(y);
          }
  }
  if ((int)cx.size() > CEM_MAX_CORNERS) return -1;
  d.n_corners = (int)cx.size();
  for (int a = 0; a < d.n_corners; ++a) {
    d.corner[a][0] = (float)cx[a];
    d.corner[a][1] = (float)cy[a];
    d.corner_vis[a] = 0;
  }
  for (int a = 0; a < d.n_corners; ++a)
    for (int b = a + 1; b < d.n_corners; ++b) {
      bool vis = true;
      for (int q = 0; q < nf && vis; ++q) vis = !host_crosses(fp[q], cx[a], cy[a], cx[b], cy[b]);
      if (vis) {
        d.corner_vis[a] |= 1ull << b;
        d.corner_vis[b] |= 1ull << a;
      }
    }
  return d.n_corners;
}

// the planner of the rollout, one query (for cem_base_path)
__global__ void base_path_kernel(const DevScene* __restrict__ s, float sx, float sy, float gx, float gy, float* xy,
                                 int* n) {
  float wx[kMaxWaypoints], wy[kMaxWaypoints];
  const int k = plan_base_path(*s, sx, sy, gx, gy, wx, wy);
  for (int i = 0; i < k; ++i) {
    xy[2 * i] = wx[i];
    xy[2 * i + 1] = wy[i];
  }
  *n = k;
}

int validate(const cem_scene_desc* s, const cem_skeleton_desc* k) {
  if (!s || !k) return fail(CEM_ERR_INVALID_ARG, "scene and skeleton descriptors are required");
  if (s->kind < CEM_SCENE_QUADRATIC || s->kind > CEM_SCENE_PICKPLACE) return fail(CEM_ERR_INVALID_ARG, "unknown scene kind");
  if (k->D < 1 || k->D > CEM_MAX_D) return fail(CEM_ERR_UNSUPPORTED, "D must be in 1..18");
  if (s->T < 1 || s->T > 1000000) return fail(CEM_ERR_UNSUPPORTED, "T must be in 1..1e6");
  if (!(s->dt > 0.0f) || !std::isfinite(s->dt)) return fail(CEM_ERR_INVALID_ARG, "dt must be positive");
  for (int d = 0; d < k->D; ++d)
    if (!(k->lo[d] <= k->hi[d]) || !std::isfinite(k->lo[d]) || !std::isfinite(k->hi[d]))
      return fail(CEM_ERR_INVALID_ARG, "bounds must be finite with lo <= hi");
  if (s->kind == CEM_SCENE_QUADRATIC) return CEM_OK;
  if (k->n_actions < 1 || k->n_actions > CEM_MAX_ACTIONS) return fail(CEM_ERR_UNSUPPORTED, "1..6 actions supported");
  int off = 0;
  for (int i = 0; i < k->n_actions; ++i) {
    const cem_action_desc& a = k->action[i];
    if (a.kind < CEM_ACT_MOVE || a.kind > CEM_ACT_PLACE) return fail(CEM_ERR_INVALID_ARG, "unknown action kind");
    const bool planar = s->kind != CEM_SCENE_PICKPLACE;
    if (planar && !(a.kind == CEM_ACT_MOVE || a.kind == CEM_ACT_PUSH))
      return fail(CEM_ERR_INVALID_ARG, "planar scenes take moveTo/push actions only");
    if (!planar && a.kind == CEM_ACT_PUSH) return fail(CEM_ERR_INVALID_ARG, "pick-place takes no push action");
    if (a.theta_offset != off) return fail(CEM_ERR_INVALID_ARG, "theta slices must be contiguous and in order");
    if (a.init_region != 0 && a.init_region != 1) return fail(CEM_ERR_INVALID_ARG, "init_region must be 0 or 1");
    if (a.init_region == 1) {
      if (a.kind != CEM_ACT_MOVE) return fail(CEM_ERR_INVALID_ARG, "only moveTo goals take an annulus region");
      if (!(a.region[2] >= 0.0f && a.region[3] > a.region[2]) || !std::isfinite(a.region[0]) ||
          !std::isfinite(a.region[1]) || !std::isfinite(a.region[3]))
        return fail(CEM_ERR_INVALID_ARG, "annulus needs finite centre and 0 <= inner < outer radius");
    }
    off += action_width(a.kind);
  }
  if (off != k->D) return fail(CEM_ERR_INVALID_ARG, "theta slices do not cover D");
  if (s->kind == CEM_SCENE_PUSH && (k->n_actions > 2))
    return fail(CEM_ERR_UNSUPPORTED, "push scenes have at most 2 actions");
  if (s->n_geoms < 0 || s->n_geoms > CEM_MAX_GEOMS) return fail(CEM_ERR_UNSUPPORTED, "at most 16 geometries");
  for (int g = 0; g < s->n_geoms; ++g)
    if (s->geom[g].n_slabs < 0 || s->geom[g].n_slabs > CEM_MAX_SLABS)
      return fail(CEM_ERR_UNSUPPORTED, "at most 6 slabs per geometry");
  if (!(s->base_mass > 0.0f)) return fail(CEM_ERR_INVALID_ARG, "base mass must be positive");
  if (s->kind == CEM_SCENE_PUSH && !(s->block_mass > 0.0f)) return fail(CEM_ERR_INVALID_ARG, "block mass must be positive");
  if (s->kind == CEM_SCENE_PICKPLACE && !(s->obj_mass > 0.0f && s->arm_l1 > 0.0f && s->arm_l2 > 0.0f))
    return fail(CEM_ERR_INVALID_ARG, "object mass and arm links must be positive");
  if (s->base_controller != 0 && s->base_controller != 1) return fail(CEM_ERR_INVALID_ARG, "base_controller is 0 or 1");
  if (s->base_controller == 1) {
    if (s->kind != CEM_SCENE_PICKPLACE) return fail(CEM_ERR_INVALID_ARG, "the A* base controller is for pick-place");
    if (!(s->base_inflate >= 0.0f) || !(s->wp_switch > 0.0f) || !(s->pid_ki >= 0.0f) || !(s->pid_irad >= 0.0f) ||
        !(s->pid_imax >= 0.0f) || !std::isfinite(s->base_inflate + s->wp_switch + s->pid_ki + s->pid_irad + s->pid_imax))
      return fail(CEM_ERR_INVALID_ARG, "A* controller: inflate, integral gain/radius/limit >= 0, switch radius > 0");
    DevScene tmp;
    if (build_base_graph(*s, tmp) < 0) return fail(CEM_ERR_UNSUPPORTED, "more than 48 planner corners");
  }
  return CEM_OK;
}

DevScene prepare(const cem_scene_desc& s, const cem_skeleton_desc& k) {
  DevScene d;
  std::memset(&d, 0, sizeof(d));
  d.kind = s.kind;
  d.T = s.T;
  d.cost_step = s.cost_mode == CEM_COST_STEP;
  d.D = k.D;
  d.n_act = s.kind == CEM_SCENE_QUADRATIC ? 0 : k.n_actions;
  d.n_geoms = s.n_geoms;
  d.goal_obj_region = s.goal_obj_region;
  d.goal_obj_held = s.goal_obj_held;
  d.goal_base_region = s.goal_base_region;
  d.dt = s.dt;
  d.g = s.g;
  d.eps = s.eps;
  d.k_contact = s.k_contact;
  d.c_contact = s.c_contact;
  d.contact_mu = s.contact_mu;
  d.force_limit = s.force_limit;
  d.w_time = s.w_time;
  d.w_goal = s.w_goal;
  d.w_viol = s.w_viol;
  d.w_obj = s.w_obj;
  d.w_base = s.w_base;
  const double dt = s.dt, g = s.g;
  // base
  d.bhx = s.base_half[0];
  d.bhy = s.base_half[1];
  d.mb = s.base_mass;
  const double Ib = s.base_mass * (4.0 * s.base_half[0] * s.base_half[0] + 4.0 * s.base_half[1] * s.base_half[1]) / 12.0;
  d.Ib = (float)Ib;
  d.dt_mb = (float)(dt / s.base_mass);
  d.dt_Ib = Ib > 0 ? (float)(dt / Ib) : 0.0f;
  d.base_cap = (float)(s.base_mu * g * dt);
  if (Ib > 0 && s.base_half[0] > 0 && s.base_half[1] > 0)
    d.base_wcap = (float)(s.base_mu * s.base_mass * g * mean_radius(s.base_half[0], s.base_half[1]) * dt / Ib);
  d.yaw_kp = s.yaw_kp;
  d.yaw_kd = s.yaw_kd;
  for (int i = 0; i < 3; ++i) {
    d.base_start[i] = s.base_start[i];
    d.base_v0[i] = s.base_v0[i];
    d.block_start[i] = s.block_start[i];
    d.block_v0[i] = s.block_v0[i];
    d.goal_center[i] = s.goal_center[i];
    d.goal_half[i] = s.goal_half[i];
    d.obj_start[i] = s.obj_start[i];
    d.obj_v0[i] = s.obj_v0[i];
    d.obj_region_c[i] = s.obj_region_c[i];
    d.obj_region_h[i] = s.obj_region_h[i];
    d.base_region_c[i] = s.base_region_c[i];
    d.base_region_h[i] = s.base_region_h[i];
  }
  // block
  d.khx = s.block_half[0];
  d.khy = s.block_half[1];
  d.mk = s.block_mass;
  if (s.block_mass > 0) {
    const double Ik = s.block_mass * (4.0 * s.block_half[0] * s.block_half[0] + 4.0 * s.block_half[1] * s.block_half[1]) / 12.0;
    d.Ik = (float)Ik;
    d.dt_mk = (float)(dt / s.block_mass);
    d.dt_Ik = (float)(dt / Ik);
    d.block_cap = (float)(s.block_mu * g * dt);
    d.block_wcap = (float)(s.block_mu * s.block_mass * g * mean_radius(s.block_half[0], s.block_half[1]) * dt / Ik);
  }
  // pick-place
  d.oh = s.obj_half;
  d.mo = s.obj_mass;
  d.obj_mu = s.obj_mu;
  d.dt_mo = s.obj_mass > 0 ? (float)(dt / s.obj_mass) : 0.0f;
  d.obj_cap = (float)(s.obj_mu * dt);
  d.arm_l1 = s.arm_l1;
  d.arm_l2 = s.arm_l2;
  d.arm_z = s.arm_z;
  d.arm_kp = s.arm_kp;
  d.arm_kd = s.arm_kd;
  d.arm_home[0] = s.arm_home[0];
  d.arm_home[1] = s.arm_home[1];
  d.grasp_reach = s.grasp_reach;
  d.grasp_kp = s.grasp_kp;
  d.grip_tol = s.grip_tol;
  // skeleton
  for (int i = 0; i < CEM_MAX_ACTIONS && i < k.n_actions; ++i) {
    d.act_kind[i] = k.action[i].kind;
    d.act_off[i] = k.action[i].theta_offset;
    d.act_ref[i] = k.action[i].success_ref;
    for (int j = 0; j < 3; ++j) d.act_nom[i][j] = k.action[i].nominal[j];
    d.act_yaw[i] = k.action[i].yaw;
    d.act_region[i] = k.action[i].init_region;
    for (int j = 0; j < 4; ++j) d.act_ring[i][j] = k.action[i].region[j];
  }
  for (int i = 0; i < k.D; ++i) {
    d.lo[i] = k.lo[i];
    d.hi[i] = k.hi[i];
  }
  for (int gi = 0; gi < s.n_geoms; ++gi) {
    d.geom_nslab[gi] = s.geom[gi].n_slabs;
    d.geom_flags[gi] = (s.geom[gi].collide_base ? 1 : 0) | (s.geom[gi].collide_object ? 2 : 0);
    int nb = 0;
    for (int si = 0; si < s.geom[gi].n_slabs; ++si) {
      const cem_slab& sl = s.geom[gi].slab[si];
      for (int j = 0; j < 3; ++j) d.slab[gi][si][j] = sl.n[j];
      d.slab[gi][si][3] = sl.lo;
      d.slab[gi][si][4] = sl.hi;
      // the movers' supports along n folded in (pick-and-place contacts)
      const double ro = (double)s.obj_half * (std::fabs((double)sl.n[0]) + std::fabs((double)sl.n[1]) +
                                              std::fabs((double)sl.n[2]));
      for (int j = 0; j < 3; ++j) d.oslab[gi][si][j] = sl.n[j];
      d.oslab[gi][si][3] = (float)((double)sl.lo - ro);
      d.oslab[gi][si][4] = (float)((double)sl.hi + ro);
      if (sl.n[2] == 0.0f) {
        const double rb = (double)s.base_half[0] * std::fabs((double)sl.n[0]) +
                          (double)s.base_half[1] * std::fabs((double)sl.n[1]);
        d.bslab[gi][nb][0] = sl.n[0];
        d.bslab[gi][nb][1] = sl.n[1];
        d.bslab[gi][nb][2] = (float)((double)sl.lo - rb);
        d.bslab[gi][nb][3] = (float)((double)sl.hi + rb);
        ++nb;
      }
    }
    d.bslab_n[gi] = nb;
  }
  // a projection on n changes by at most max |n_i| per metre of path (1 for
  // the unit normals the descriptor asks for)
  float nmax = 1.0f;
  for (int gi = 0; gi < s.n_geoms; ++gi)
    for (int si = 0; si < s.geom[gi].n_slabs; ++si)
      for (int j = 0; j < 3; ++j) {
        const float a = std::fabs(s.geom[gi].slab[si].n[j]);
        nmax = a <= nmax ? nmax : a;
      }
  d.sep_scale = std::isfinite(nmax) ? 1.0f / nmax : 0.0f;
  for (int i = 0; i < CEM_MAX_D; ++i) d.theta_star[i] = s.theta_star[i];
  for (int i = 0; i < k.D * k.D; ++i) d.A[i] = s.A[i];
  if (s.kind == CEM_SCENE_PICKPLACE && s.base_controller == 1) {
    d.base_ctrl = 1;
    d.base_infl = s.base_inflate;
    d.wp_switch = s.wp_switch;
    d.pid_ki = s.pid_ki;
    d.pid_irad = s.pid_irad;
    d.pid_imax = s.pid_imax;
    build_base_graph(s, d);
  }
  return d;
}

int default_block(const cem_ctx* h, int N) {
  if (h->block > 0) return h->block;
  return cem::default_rollout_block(N, h->host.kind, h->tpr, h->dr_on ? h->dr.M : 1);
}

// byte offsets of the solve state block (iters: history capacity)
struct StateLayout {
  size_t track, status, keff, mean, cov, chol, hist_J, hist_keff, hist_cnt, end;
};

StateLayout state_layout(int iters) {
  auto up16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
  StateLayout L;
  size_t o = 0;
  L.track = o;
  o = up16(o + sizeof(Track));
  L.status = o;
  o = up16(o + sizeof(int32_t));
  L.keff = o;
  o = up16(o + sizeof(int32_t));
  L.mean = o;
  o = up16(o + sizeof(float) * CEM_MAX_D);
  L.cov = o;
  o = up16(o + sizeof(float) * CEM_MAX_D * CEM_MAX_D);
  L.chol = o;
  o = up16(o + sizeof(float) * CEM_MAX_D * CEM_MAX_D);
  L.hist_J = o;
  o = up16(o + sizeof(float) * (size_t)iters);
  L.hist_keff = o;
  o = up16(o + sizeof(int32_t) * (size_t)iters);
  L.hist_cnt = o;
  o = up16(o + sizeof(int32_t) * 4 * (size_t)iters);
  L.end = o;
  return L;
}

void free_work(cem_ctx* h) {
  cudaFree(h->theta_d);
  cudaFree(h->J_d);
  cudaFree(h->cls_d);
  cudaFree(h->state_d);
  cudaFreeHost(h->state_h);
  h->state_d = h->state_h = nullptr;
  h->theta_d = nullptr;
  h->J_d = nullptr;
  h->cls_d = nullptr;
  h->mean_d = h->cov_d = h->chol_d = nullptr;
  h->keff_d = h->status_d = nullptr;
  h->track_d = nullptr;
  h->hist_J_d = nullptr;
  h->hist_keff_d = nullptr;
  h->hist_cnt_d = nullptr;
  h->cap_N = h->cap_K = h->cap_iters = 0;
}

int ensure_work(cem_ctx* h, int N, int iters) {
  const int D = h->skel.D;
  if (N <= h->cap_N && iters <= h->cap_iters && h->mean_d) return CEM_OK;
  if (h->graph) {
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  free_work(h);
  const int n = N > 0 ? N : 1, it = iters > 0 ? iters : 1;
  const StateLayout L = state_layout(it);
  if (dev_malloc(&h->theta_d, sizeof(float) * (size_t)n * D) != cudaSuccess ||
      dev_malloc(&h->J_d, sizeof(float) * (size_t)n) != cudaSuccess ||
      dev_malloc(&h->cls_d, (size_t)n) != cudaSuccess || dev_malloc(&h->state_d, L.end) != cudaSuccess ||
      cudaMallocHost(&h->state_h, L.end) != cudaSuccess) {
    cudaGetLastError();
    free_work(h);
    return fail(CEM_ERR_NO_MEMORY, "allocation of the solve workspace failed");
  }
  h->track_d = reinterpret_cast<Track*>(h->state_d + L.track);
  h->status_d = reinterpret_cast<int32_t*>(h->state_d + L.status);
  h->keff_d = reinterpret_cast<int32_t*>(h->state_d + L.keff);
  h->mean_d = reinterpret_cast<float*>(h->state_d + L.mean);
  h->cov_d = reinterpret_cast<float*>(h->state_d + L.cov);
  h->chol_d = reinterpret_cast<float*>(h->state_d + L.chol);
  h->hist_J_d = reinterpret_cast<float*>(h->state_d + L.hist_J);
  h->hist_keff_d = reinterpret_cast<int32_t*>(h->state_d + L.hist_keff);
  h->hist_cnt_d = reinterpret_cast<int32_t*>(h->state_d + L.hist_cnt);
  h->cap_N = n;
  h->cap_iters = it;
  return CEM_OK;
}

RefitArgs refit_args(const cem_ctx* h, const float* theta, const float* J, const uint8_t* cls, int N, int K,
                     int cov_mode) {
  RefitArgs a;
  std::memset(&a, 0, sizeof(a));
  a.theta = theta;
  a.J = J;
  a.cls = cls;
  a.N = N;
  a.D = h->skel.D;
  a.K = K;
  a.cov_mode = cov_mode;
  for (int d = 0; d < h->skel.D; ++d) {
    a.lo[d] = h->skel.lo[d];
    a.hi[d] = h->skel.hi[d];
  }
  return a;
}

// one CE iteration on h->stream: sample -> rollout -> refit (reads and
// advances the device-side iteration counter)
// the handle's randomisation for one launch: environments of the device
// loop's current iteration (iter_ptr) or of iteration `iter`
const DrArgs* dr_for(cem_ctx* h, DrArgs& tmp, uint32_t problem, const uint32_t* iter_ptr, uint32_t iter) {
  if (!h->dr_on) return nullptr;
  tmp = h->dr;
  tmp.problem = problem;
  tmp.iter = iter;
  tmp.iter_ptr = iter_ptr;
  return &tmp;
}

cudaError_t enqueue_iteration(cem_ctx* h, uint64_t seed, uint32_t problem, int N, int K, int cov_mode) {
  cudaError_t e = launch_sample(h->mean_d, h->chol_d, seed, &h->track_d->iter, 0, problem, N, h->skel.D, h->theta_d,
                                h->stream);
  if (e != cudaSuccess) return e;
  DrArgs tmp;
  e = launch_rollout(h->scene_d, h->host.kind, h->theta_d, N, h->J_d, h->cls_d, default_block(h, N), h->tpr,
                     dr_for(h, tmp, problem, &h->track_d->iter, 0), h->stream, h->host.base_ctrl != 0);
  if (e != cudaSuccess) return e;
  RefitArgs a = refit_args(h, h->theta_d, h->J_d, h->cls_d, N, K, cov_mode);
  a.mean = h->mean_d;
  a.cov = h->cov_d;
  a.chol = h->chol_d;
  a.k_eff = h->keff_d;
  a.track = h->track_d;
  a.hist_J = h->hist_J_d;
  a.hist_keff = h->hist_keff_d;
  a.hist_cnt = h->hist_cnt_d;
  a.status = h->status_d;
  return launch_refit(a, h->stream);
}

}  // namespace

namespace cem {
const cem_skeleton_desc& handle_skeleton(cem_handle h) { return h->skel; }

int handle_solve_buffers(cem_handle h, int N, int iters, SolveBuffers* b) {
  int rc = ensure_work(h, N, iters);
  if (rc != CEM_OK) return rc;
  b->theta = h->theta_d;
  b->J = h->J_d;
  b->cls = h->cls_d;
  b->mean = h->mean_d;
  b->cov = h->cov_d;
  b->chol = h->chol_d;
  b->keff = h->keff_d;
  b->status = h->status_d;
  b->track = h->track_d;
  b->hist_J = h->hist_J_d;
  b->hist_keff = h->hist_keff_d;
  b->hist_cnt = h->hist_cnt_d;
  b->stream = h->stream;
  b->ev0 = h->ev0;
  b->ev1 = h->ev1;
  b->scene = h->scene_d;
  b->kind = h->host.kind;
  b->astar = h->host.base_ctrl != 0;
  b->block = default_block(h, N);
  b->tpr = h->tpr;
  b->dr = h->dr_on ? &h->dr : nullptr;
  return CEM_OK;
}

int handle_init_distribution(cem_handle h, const cem_solve_params* p, SolveBuffers* b) {
  const int D = h->skel.D;
  std::vector<float> mean(D), cov((size_t)D * D, 0.0f), chol((size_t)D * D, 0.0f);
  for (int d = 0; d < D; ++d) {
    mean[d] = p->init_mean_h ? p->init_mean_h[d] : 0.5f * (h->skel.lo[d] + h->skel.hi[d]);
    if (!p->init_cov_h) cov[d * D + d] = std::pow(0.25f * (h->skel.hi[d] - h->skel.lo[d]), 2.0f);
  }
  if (p->init_cov_h)
    for (int i = 0; i < D * D; ++i) cov[i] = p->init_cov_h[i];
  if (p->init_chol_h) {  // a resumed run: the sampler's exact state
    for (int i = 0; i < D * D; ++i) chol[i] = p->init_chol_h[i];
  } else {  // host Cholesky of the initial covariance (FP64)
    std::vector<double> L((size_t)D * D, 0.0);
    for (int j = 0; j < D; ++j) {
      double s = cov[j * D + j];
      for (int k = 0; k < j; ++k) s -= L[j * D + k] * L[j * D + k];
      if (!(s > 0.0)) return fail(CEM_ERR_NOT_PD, "initial covariance is not positive definite");
      L[j * D + j] = std::sqrt(s);
      for (int i = j + 1; i < D; ++i) {
        double t = cov[i * D + j];
        for (int k = 0; k < j; ++k) t -= L[i * D + k] * L[j * D + k];
        L[i * D + j] = t / L[j * D + j];
      }
    }
    for (int i = 0; i < D * D; ++i) chol[i] = (float)L[i];
  }
  Track tr;
  std::memset(&tr, 0, sizeof(tr));
  tr.iter = p->start_iter;
  tr.base_iter = p->start_iter;
  tr.best_cls = 4;
  tr.best_J = INFINITY;
  tr.hist_len = p->iters;
  const int32_t zero = 0;
  // the pinned mirror takes the initial state; one copy moves it
  const StateLayout L = state_layout(h->cap_iters);
  unsigned char* m = h->state_h;
  CEM_CUDA(cudaStreamSynchronize(b->stream));  // nothing of an earlier call still reads or fills the mirror
  std::memcpy(m + L.track, &tr, sizeof(Track));
  std::memcpy(m + L.status, &zero, sizeof(int32_t));
  std::memcpy(m + L.mean, mean.data(), sizeof(float) * D);
  std::memcpy(m + L.cov, cov.data(), sizeof(float) * D * D);
  std::memcpy(m + L.chol, chol.data(), sizeof(float) * D * D);
  CEM_CUDA(cudaMemcpyAsync(h->state_d, m, L.hist_J, cudaMemcpyHostToDevice, b->stream));
  return CEM_OK;
}

int handle_read_result(cem_handle h, const cem_solve_params* p, SolveBuffers* b, cem_result* out) {
  const int D = h->skel.D;
  Track tr;
  int32_t status = 0;
  // the state block (and the histories asked for) into the pinned mirror,
  // one copy per contiguous range, then one synchronisation
  const StateLayout L = state_layout(h->cap_iters);
  unsigned char* m = h->state_h;
  const size_t n_j = p->best_J_hist_h ? sizeof(float) * (size_t)p->iters : 0;
  CEM_CUDA(cudaMemcpyAsync(m, h->state_d, L.hist_J + n_j, cudaMemcpyDeviceToHost, b->stream));
  if (p->k_eff_hist_h)
    CEM_CUDA(cudaMemcpyAsync(m + L.hist_keff, h->state_d + L.hist_keff, sizeof(int32_t) * (size_t)p->iters,
                             cudaMemcpyDeviceToHost, b->stream));
  if (p->class_count_hist_h)
    CEM_CUDA(cudaMemcpyAsync(m + L.hist_cnt, h->state_d + L.hist_cnt, sizeof(int32_t) * 4 * (size_t)p->iters,
                             cudaMemcpyDeviceToHost, b->stream));
  CEM_CUDA(cudaStreamSynchronize(b->stream));
  std::memcpy(&tr, m + L.track, sizeof(Track));
  std::memcpy(&status, m + L.status, sizeof(int32_t));
  std::memcpy(out->mean, m + L.mean, sizeof(float) * D);
  std::memcpy(out->cov, m + L.cov, sizeof(float) * D * D);
  std::memcpy(out->chol, m + L.chol, sizeof(float) * D * D);
  if (p->best_J_hist_h) std::memcpy(p->best_J_hist_h, m + L.hist_J, n_j);
  if (p->k_eff_hist_h) std::memcpy(p->k_eff_hist_h, m + L.hist_keff, sizeof(int32_t) * (size_t)p->iters);
  if (p->class_count_hist_h)
    std::memcpy(p->class_count_hist_h, m + L.hist_cnt, sizeof(int32_t) * 4 * (size_t)p->iters);
  float ms = 0.0f;
  CEM_CUDA(cudaEventElapsedTime(&ms, b->ev0, b->ev1));
  out->elapsed_ms = ms;
  out->D = D;
  out->iters_done = (int32_t)(tr.iter - tr.base_iter);
  out->best_J = tr.best_J;
  out->best_class = tr.best_cls;
  for (int d = 0; d < CEM_MAX_D; ++d) out->best_theta[d] = d < D ? tr.best_theta[d] : 0.0f;
  if (status != 0) return fail(CEM_ERR_NOT_PD, "covariance not positive definite after the diagonal fallback");
  return CEM_OK;
}

int validate_descriptors(const cem_scene_desc* s, const cem_skeleton_desc* k) { return validate(s, k); }
DevScene prepare_scene(const cem_scene_desc& s, const cem_skeleton_desc& k) { return prepare(s, k); }
int set_last_error(int code, const std::string& msg) { return fail(code, msg); }
int default_rollout_block(int N, int kind, int tpr, int envs) {
  // spread small batches over every SM scheduler: CTAs of 16 threads (each
  // half-warp its own warp, 4 schedulers per SM) up to one and a half warps a
  // scheduler, larger CTAs after that by the same measure, up to 128 threads.
  // Push, us with 16 / 32 / 64 threads: N = 4096 565 / 587 / 585, N = 8192 570 /
  // 596 / 584, N = 16384 625 / 599 / 586 (the rule takes 32 there; 64 is 2 %
  // faster); at N = 196,608 128 threads are 4 % faster than 256.
  // The environments of a randomised sample are rollouts of their own here:
  // 1000 push samples in 8 environments 577 / 614 / 627, 1500 576 / 617 / 619.
  int sms = 152;
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const long long R = (long long)N * envs;
  int b = 16;
  while (b < 128 && (R + b - 1) / b > 6 * sms) b *= 2;
  if (kind == CEM_SCENE_PICKPLACE && tpr == 1) {
    // pick-and-place lanes spend long stretches in different actions, so a
    // warp pays for its lanes' different branches one after another: fewer
    // lanes per warp, about 14 warps per SM (3.5 per scheduler), measured
    // 6.7 ms against 7.5 ms at N = 4096 (2 lanes) and equal at N = 16384; 3.0
    // against 3.9 ms for 256 samples in 8 environments (8 lanes, one sample's)
    const double target = (double)R / (14.0 * sms);
    int s = 2;
    while (s < 256 && s * 1.41 < target) s *= 2;
    if (s < b) b = s;
  }
  return b;
}
}  // namespace cem

namespace cem {
cudaError_t dev_malloc_bytes(void** p, size_t bytes) {
  int k = g_fail_alloc.load(std::memory_order_relaxed);
  while (k > 0) {  // count this allocation down; the one that takes the count to 0 fails
    if (g_fail_alloc.compare_exchange_weak(k, k - 1, std::memory_order_relaxed)) {
      if (k == 1) {
        *p = nullptr;
        return cudaErrorMemoryAllocation;
      }
      break;
    }
  }
  return cudaMalloc(p, bytes);
}
}  // namespace cem

extern "C" {

const char* cem_last_error(void) { return g_err.c_str(); }
const char* cem_version(void) { return "cemtamp 0.1 (sm_103a)"; }

int cem_scene_create(const cem_scene_desc* scene, const cem_skeleton_desc* skel, cem_handle* out) {
  g_err.clear();
  if (!out) return fail(CEM_ERR_INVALID_ARG, "out handle pointer is NULL");
  *out = nullptr;
  int rc = validate(scene, skel);
  if (rc != CEM_OK) return rc;
  cem_ctx* h = new cem_ctx();
  h->desc = *scene;
  h->skel = *skel;
  h->host = prepare(*scene, *skel);
  cudaError_t e = configure_refit();
  if (e == cudaSuccess) e = dev_malloc(&h->scene_d, sizeof(DevScene));
  if (e == cudaSuccess) e = cudaMemcpy(h->scene_d, &h->host, sizeof(DevScene), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking);
  if (e == cudaSuccess) e = cudaEventCreate(&h->ev0);
  if (e == cudaSuccess) e = cudaEventCreate(&h->ev1);
  if (e != cudaSuccess) {
    cudaGetLastError();
    cem_scene_destroy(h);
    return cuda_fail(e, "cem_scene_create");
  }
  *out = h;
  return CEM_OK;
}

int cem_scene_destroy(cem_handle h) {
  if (!h) return CEM_OK;
  if (h->stream) cudaStreamSynchronize(h->stream);
  if (h->graph) cudaGraphExecDestroy(h->graph);
  free_work(h);
  cudaFree(h->scene_d);
  if (h->ev0) cudaEventDestroy(h->ev0);
  if (h->ev1) cudaEventDestroy(h->ev1);
  if (h->stream) cudaStreamDestroy(h->stream);
  delete h;
  return CEM_OK;
}

int cem_set_launch(cem_handle h, int block_threads) {
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (block_threads != 0 && block_threads != 2 && block_threads != 4 && block_threads != 8 && block_threads != 16 &&
      (block_threads < 32 || block_threads > 256 || block_threads % 32))
    return fail(CEM_ERR_INVALID_ARG, "block size must be 0, 8, 16 or a multiple of 32 in 32..256");
  h->block = block_threads;
  if (h->graph) {  // a captured iteration keeps the launch shape it was built with
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  return CEM_OK;
}

int cem_set_randomization(cem_handle h, int M, float delta_mu, float delta_mass, uint64_t seed) {
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (M < 1 || M > 32 || (M & (M - 1))) return fail(CEM_ERR_INVALID_ARG, "M must be 1, 2, 4, 8, 16 or 32");
  if (!(delta_mu >= 0.0f && delta_mu < 1.0f) || !(delta_mass >= 0.0f && delta_mass < 1.0f))
    return fail(CEM_ERR_INVALID_ARG, "spreads must lie in [0, 1)");
  h->dr_on = !(M == 1 && delta_mu == 0.0f && delta_mass == 0.0f);
  h->dr = DrArgs{};
  h->dr.M = M;
  h->dr.dmu = delta_mu;
  h->dr.dm = delta_mass;
  h->dr.seed = seed;
  if (h->graph) {  // a captured iteration keeps the rollout it was built with
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  return CEM_OK;
}

int cem_set_threads_per_rollout(cem_handle h, int tpr) {
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (tpr != 1 && tpr != 8 && tpr != 32) return fail(CEM_ERR_INVALID_ARG, "threads per rollout must be 1, 8 or 32");
  h->tpr = tpr;
  if (h->graph) {
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  return CEM_OK;
}

int cem_get_launch(cem_handle h, int N, int* block_out, int* tpr_out) {
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (block_out) *block_out = default_block(h, N > 0 ? N : 1);
  if (tpr_out) *tpr_out = h->host.kind == CEM_SCENE_PICKPLACE ? h->tpr : 1;
  return CEM_OK;
}

int cem_sample(cem_handle h, const float* mean_d, const float* chol_d, uint64_t seed, uint32_t iter, uint32_t problem,
               int N, float* theta_d, void* stream) {
  g_err.clear();
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (N < 0 || N > CEM_MAX_N) return fail(CEM_ERR_UNSUPPORTED, "N must be in 0..2^20");
  if (N == 0) return CEM_OK;
  if (!is_device_ptr(mean_d) || !is_device_ptr(chol_d) || !is_device_ptr(theta_d))
    return fail(CEM_ERR_INVALID_ARG, "mean, chol and theta must be device pointers");
  cudaError_t e = launch_sample(mean_d, chol_d, seed, nullptr, iter, problem, N, h->skel.D, theta_d,
                                (cudaStream_t)stream);
  return e == cudaSuccess ? CEM_OK : cuda_fail(e, "cem_sample");
}

int cem_philox_words(cem_handle h, uint64_t seed, uint32_t iter, uint32_t problem, int N, uint32_t* words_d,
                     void* stream) {
  g_err.clear();
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (N < 0 || N > CEM_MAX_N) return fail(CEM_ERR_UNSUPPORTED, "N must be in 0..2^20");
  if (N == 0) return CEM_OK;
  if (!is_device_ptr(words_d)) return fail(CEM_ERR_INVALID_ARG, "words must be a device pointer");
  cudaError_t e = launch_philox_words(seed, iter, problem, N, h->skel.D, words_d, (cudaStream_t)stream);
  return e == cudaSuccess ? CEM_OK : cuda_fail(e, "cem_philox_words");
}

int cem_rollout_batch(cem_handle h, const float* theta_d, int N, float* J_d, uint8_t* cls_d, void* stream) {
  g_err.clear();
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (N < 0 || N > CEM_MAX_N) return fail(CEM_ERR_UNSUPPORTED, "N must be in 0..2^20");
  if (N == 0) return CEM_OK;
  if (!is_device_ptr(theta_d) || !is_device_ptr(J_d) || !is_device_ptr(cls_d))
    return fail(CEM_ERR_INVALID_ARG, "theta, J and cls must be device pointers");
  DrArgs tmp;
  cudaError_t e = launch_rollout(h->scene_d, h->host.kind, theta_d, N, J_d, cls_d, default_block(h, N), h->tpr,
                                 dr_for(h, tmp, 0, nullptr, 0),
                                 (cudaStream_t)stream, h->host.base_ctrl != 0);
  return e == cudaSuccess ? CEM_OK : cuda_fail(e, "cem_rollout_batch");
}

int cem_rollout_trace(cem_handle h, const float* theta_d, int N, int steps, float* states_d, void* stream) {
  g_err.clear();
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (N < 0 || N > 65536 || steps < 0 || steps > 100000) return fail(CEM_ERR_UNSUPPORTED, "trace: N <= 65536, steps <= 1e5");
  if (N == 0 || steps == 0) return CEM_OK;
  if (h->host.kind == CEM_SCENE_QUADRATIC) return fail(CEM_ERR_UNSUPPORTED, "quadratic scenes have no state");
  if (!is_device_ptr(theta_d) || !is_device_ptr(states_d))
    return fail(CEM_ERR_INVALID_ARG, "theta and states must be device pointers");
  cudaError_t e = launch_trace(h->scene_d, h->host.kind, theta_d, N, steps, states_d, (cudaStream_t)stream,
                               h->host.base_ctrl != 0);
  return e == cudaSuccess ? CEM_OK : cuda_fail(e, "cem_rollout_trace");
}

int cem_refit(cem_handle h, const float* theta_d, const float* J_d, const uint8_t* cls_d, int N, int K, int cov_mode,
              float* mean_d, float* cov_d, float* chol_d, int32_t* elite_idx_d, int32_t* k_eff_d, void* stream) {
  g_err.clear();
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (N < 0 || N > CEM_MAX_N) return fail(CEM_ERR_UNSUPPORTED, "N must be in 0..2^20");
  if (K < 1 || K > CEM_MAX_K) return fail(CEM_ERR_UNSUPPORTED, "K must be in 1..4096");
  if (cov_mode != CEM_COV_FULL && cov_mode != CEM_COV_DIAG) return fail(CEM_ERR_INVALID_ARG, "unknown cov mode");
  if (!is_device_ptr(mean_d) || !is_device_ptr(cov_d) || !is_device_ptr(chol_d))
    return fail(CEM_ERR_INVALID_ARG, "mean, cov and chol must be device pointers");
  if (N > 0 && (!is_device_ptr(theta_d) || !is_device_ptr(J_d) || !is_device_ptr(cls_d)))
    return fail(CEM_ERR_INVALID_ARG, "theta, J and cls must be device pointers");
  if ((elite_idx_d && !is_device_ptr(elite_idx_d)) || (k_eff_d && !is_device_ptr(k_eff_d)))
    return fail(CEM_ERR_INVALID_ARG, "elite_idx and k_eff must be device pointers or NULL");
  RefitArgs a = refit_args(h, theta_d, J_d, cls_d, N, K, cov_mode);
  a.mean = mean_d;
  a.cov = cov_d;
  a.chol = chol_d;
  a.elite_idx = elite_idx_d;
  a.k_eff = k_eff_d;
  cudaError_t e = launch_refit(a, (cudaStream_t)stream);
  return e == cudaSuccess ? CEM_OK : cuda_fail(e, "cem_refit");
}

int cem_solve(cem_handle h, const cem_solve_params* p, cem_result* out) {
  g_err.clear();
  if (!h || !p || !out) return fail(CEM_ERR_INVALID_ARG, "null argument");
  if (p->N < 1 || p->N > CEM_MAX_N) return fail(CEM_ERR_UNSUPPORTED, "N must be in 1..2^20");
  if (p->K < 1 || p->K > CEM_MAX_K) return fail(CEM_ERR_UNSUPPORTED, "K must be in 1..4096");
  if (p->iters < 1 || p->iters > 100000) return fail(CEM_ERR_UNSUPPORTED, "iters must be in 1..1e5");
  if (p->cov_mode != CEM_COV_FULL && p->cov_mode != CEM_COV_DIAG) return fail(CEM_ERR_INVALID_ARG, "unknown cov mode");
  SolveBuffers b;
  int rc = cem::handle_solve_buffers(h, p->N, p->iters, &b);
  if (rc != CEM_OK) return rc;
  rc = cem::handle_init_distribution(h, p, &b);
  if (rc != CEM_OK) return rc;
  if (p->use_graph) {
    const bool stale = !h->graph || h->graph_N != p->N || h->graph_K != p->K || h->graph_cov != p->cov_mode ||
                       h->graph_seed != p->seed || h->graph_problem != p->problem;
    if (stale) {
      if (h->graph) {
        cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
      }
      cudaGraph_t g;
      CEM_CUDA(cudaStreamBeginCapture(h->stream, cudaStreamCaptureModeThreadLocal));
      cudaError_t e = enqueue_iteration(h, p->seed, p->problem, p->N, p->K, p->cov_mode);
      cudaError_t e2 = cudaStreamEndCapture(h->stream, &g);
      if (e != cudaSuccess) return cuda_fail(e, "capture of the CE iteration");
      if (e2 != cudaSuccess) return cuda_fail(e2, "cudaStreamEndCapture");
      e = cudaGraphInstantiate(&h->graph, g, 0);
      cudaGraphDestroy(g);
      if (e != cudaSuccess) return cuda_fail(e, "cudaGraphInstantiate");
      h->graph_N = p->N;
      h->graph_K = p->K;
      h->graph_cov = p->cov_mode;
      h->graph_seed = p->seed;
      h->graph_problem = p->problem;
    }
  }
  CEM_CUDA(cudaEventRecord(h->ev0, h->stream));
  for (int j = 0; j < p->iters; ++j) {
    if (p->use_graph) {
      CEM_CUDA(cudaGraphLaunch(h->graph, h->stream));
    } else {
      cudaError_t e = enqueue_iteration(h, p->seed, p->problem, p->N, p->K, p->cov_mode);
      if (e != cudaSuccess) return cuda_fail(e, "CE iteration");
    }
  }
  CEM_CUDA(cudaEventRecord(h->ev1, h->stream));
  return cem::handle_read_result(h, p, &b, out);
}

int cem_base_path(cem_handle h, float sx, float sy, float gx, float gy, float* xy_h, int cap, int* n_out) {
  g_err.clear();
  if (!h || !n_out) return fail(CEM_ERR_INVALID_ARG, "null argument");
  if (!h->host.base_ctrl) return fail(CEM_ERR_UNSUPPORTED, "the scene has no A* base controller");
  if (cap < 0 || (cap > 0 && !xy_h)) return fail(CEM_ERR_INVALID_ARG, "cap >= 0 and an output array");
  float* buf = nullptr;
  int* cnt = nullptr;
  CEM_CUDA(dev_malloc(&buf, sizeof(float) * 2 * kMaxWaypoints));
  cudaError_t e = dev_malloc(&cnt, sizeof(int));
  if (e == cudaSuccess) {
    base_path_kernel<<<1, 1, 0, h->stream>>>(h->scene_d, sx, sy, gx, gy, buf, cnt);
    e = cudaGetLastError();
  }
  float out[2 * kMaxWaypoints];
  int n = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&n, cnt, sizeof(int), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(out, buf, sizeof(out), cudaMemcpyDeviceToHost, h->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
  cudaFree(buf);
  cudaFree(cnt);
  if (e != cudaSuccess) return cuda_fail(e, "cem_base_path");
  for (int i = 0; i < 2 * std::min(n, cap); ++i) xy_h[i] = out[i];
  *n_out = n;
  return CEM_OK;
}

int cem_debug_status(int* code_out, int reset) {
  if (!code_out) return fail(CEM_ERR_INVALID_ARG, "cem_debug_status: code_out is NULL");
  *code_out = 0;
#ifdef CEM_DEBUG
  int c[4] = {0, 0, 0, 0};  // rollout.cu (rollouts, orders), refit.cu, surrogate.cu (screening), mlp_train.cu
  cudaError_t e = cudaDeviceSynchronize();
  if (e == cudaSuccess) e = debug_status_rollout(&c[0], reset != 0);
  if (e == cudaSuccess) e = debug_status_refit(&c[1], reset != 0);
  if (e == cudaSuccess) e = debug_status_surrogate(&c[2], reset != 0);
  if (e == cudaSuccess) e = debug_status_train(&c[3], reset != 0);
  if (e != cudaSuccess) return cuda_fail(e, "cem_debug_status");
  *code_out = c[0] ? c[0] : c[1] ? c[1] : c[2] ? c[2] : c[3];
  return CEM_OK;
#else
  (void)reset;
  return fail(CEM_ERR_UNSUPPORTED, "cem_debug_status: a release build (no bounds checks)");
#endif
}

int cem_test_fail_allocation(int k) {
  if (k < 0) return fail(CEM_ERR_INVALID_ARG, "cem_test_fail_allocation: k must be >= 0");
  g_fail_alloc.store(k, std::memory_order_relaxed);
  return CEM_OK;
}

int cem_debug_selftest(void) {
#ifdef CEM_DEBUG
  const cudaError_t e = debug_selftest_rollout();
  return e == cudaSuccess ? CEM_OK : cuda_fail(e, "cem_debug_selftest");
#else
  return fail(CEM_ERR_UNSUPPORTED, "cem_debug_selftest: a release build (no bounds checks)");
#endif
}

int cem_n_env(int n0, int n1, int j1, int j) {
  if (j1 <= 0) return j <= 0 ? n0 : n1;
  if (j >= j1) return n1;
  if (j <= 0) return n0;
  // n0 + (n1 - n0) j / j1 = num / j1 > 0, rounded half up in integers
  const long long num = (long long)n0 * j1 + (long long)(n1 - n0) * j;
  return (int)((2 * num + j1) / (2LL * j1));
}

int cem_sample_uniform(cem_handle h, uint64_t seed, uint32_t problem, int N, float* theta_d, void* stream) {
  g_err.clear();
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (N < 0 || N > CEM_MAX_N) return fail(CEM_ERR_UNSUPPORTED, "N must be in 0..2^20");
  if (N == 0) return CEM_OK;
  if (!is_device_ptr(theta_d)) return fail(CEM_ERR_INVALID_ARG, "theta must be a device pointer");
  cudaError_t e = launch_sample_uniform(h->scene_d, seed, problem, N, h->skel.D, theta_d, (cudaStream_t)stream);
  return e == cudaSuccess ? CEM_OK : cuda_fail(e, "cem_sample_uniform");
}

int cem_solve_paper(cem_handle h, const cem_paper_params* p, cem_result* out) {
  g_err.clear();
  if (!h || !p || !out) return fail(CEM_ERR_INVALID_ARG, "null argument");
  if (p->n0 < 1 || p->n0 > CEM_MAX_N || p->n1 < 1 || p->n1 > CEM_MAX_N || p->j1 < 0)
    return fail(CEM_ERR_UNSUPPORTED, "n0, n1 must be in 1..2^20 and j1 >= 0");
  if (p->K < 1 || p->K > CEM_MAX_K) return fail(CEM_ERR_UNSUPPORTED, "K must be in 1..4096");
  if (p->iters < 1 || p->iters > 100000) return fail(CEM_ERR_UNSUPPORTED, "iters must be in 1..1e5");
  if (p->cov_mode != CEM_COV_FULL && p->cov_mode != CEM_COV_DIAG) return fail(CEM_ERR_INVALID_ARG, "unknown cov mode");
  const int nmax = p->n0 > p->n1 ? p->n0 : p->n1;
  cem_solve_params q;
  std::memset(&q, 0, sizeof(q));
  q.seed = p->seed;
  q.N = nmax;
  q.K = p->K;
  q.iters = p->iters;
  q.cov_mode = p->cov_mode;
  q.problem = p->problem;
  q.best_J_hist_h = p->best_J_hist_h;
  q.k_eff_hist_h = p->k_eff_hist_h;
  q.class_count_hist_h = p->class_count_hist_h;
  SolveBuffers b;
  int rc = cem::handle_solve_buffers(h, nmax, p->iters, &b);
  if (rc != CEM_OK) return rc;
  // loop state reset; iteration 0 does not read the Gaussian (its samples are uniform)
  rc = cem::handle_init_distribution(h, &q, &b);
  if (rc != CEM_OK) return rc;
  const int D = h->skel.D;
  CEM_CUDA(cudaEventRecord(h->ev0, h->stream));
  for (int j = 0; j < p->iters; ++j) {
    const int N = cem_n_env(p->n0, p->n1, p->j1, j);
    if (p->n_env_hist_h) p->n_env_hist_h[j] = N;
    cudaError_t e = j == 0 ? launch_sample_uniform(h->scene_d, p->seed, p->problem, N, D, h->theta_d, h->stream)
                           : launch_sample(h->mean_d, h->chol_d, p->seed, &h->track_d->iter, 0, p->problem, N, D,
                                           h->theta_d, h->stream);
    DrArgs tmp;
    if (e == cudaSuccess)
      e = launch_rollout(h->scene_d, h->host.kind, h->theta_d, N, h->J_d, h->cls_d, default_block(h, N), h->tpr,
                         dr_for(h, tmp, p->problem, &h->track_d->iter, 0), h->stream, h->host.base_ctrl != 0);
    if (e == cudaSuccess) {
      RefitArgs a = refit_args(h, h->theta_d, h->J_d, h->cls_d, N, p->K, p->cov_mode);
      a.mean = h->mean_d;
      a.cov = h->cov_d;
      a.chol = h->chol_d;
      a.k_eff = h->keff_d;
      a.track = h->track_d;
      a.hist_J = h->hist_J_d;
      a.hist_keff = h->hist_keff_d;
      a.hist_cnt = h->hist_cnt_d;
      a.status = h->status_d;
      e = launch_refit(a, h->stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "paper CE iteration");
  }
  CEM_CUDA(cudaEventRecord(h->ev1, h->stream));
  return cem::handle_read_result(h, &q, &b, out);
}

int cem_autotune(cem_handle h, int N, const char* cache_path, int* block_out) {
  g_err.clear();
  if (!h) return fail(CEM_ERR_INVALID_ARG, "null handle");
  if (N < 1 || N > CEM_MAX_N) return fail(CEM_ERR_UNSUPPORTED, "N must be in 1..2^20");
  int dev = 0, sms = 0;
  CEM_CUDA(cudaGetDevice(&dev));
  CEM_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  char keybuf[256];
  std::snprintf(keybuf, sizeof(keybuf), "kind=%d T=%d D=%d A=%d G=%d N=%d sms=%d", h->host.kind, h->host.T,
                h->host.D, h->host.n_act, h->host.n_geoms, N, sms);
  const std::string key(keybuf);
  const bool multi_lane = h->host.kind == CEM_SCENE_PICKPLACE;
  if (cache_path) {  // cache lines: "<key>|<block>|<threads per rollout>"
    std::ifstream in(cache_path);
    std::string line;
    while (std::getline(in, line)) {
      const size_t bar = line.find('|');
      if (bar != std::string::npos && line.substr(0, bar) == key) {
        int b = 0, t = 1;
        const int got = std::sscanf(line.c_str() + bar + 1, "%d|%d", &b, &t);
        const bool ok_b = b == 2 || b == 4 || b == 8 || b == 16 || (b >= 32 && b <= 256 && b % 32 == 0);
        const bool ok_t = t == 1 || (multi_lane && (t == 8 || t == 32) && b >= 32);
        if (got >= 1 && ok_b && ok_t) {
          h->block = b;
          h->tpr = t;
          if (block_out) *block_out = b;
          if (h->graph) {
            cudaGraphExecDestroy(h->graph);
            h->graph = nullptr;
          }
          return CEM_OK;
        }
      }
    }
  }
  int rc = ensure_work(h, N, 1);
  if (rc != CEM_OK) return rc;
  // sample once from the initial distribution so the timed rollouts see
  // realistic parameter vectors
  const int D = h->skel.D;
  std::vector<float> mean(D), chol((size_t)D * D, 0.0f);
  for (int d = 0; d < D; ++d) {
    mean[d] = 0.5f * (h->skel.lo[d] + h->skel.hi[d]);
    chol[d * D + d] = 0.25f * (h->skel.hi[d] - h->skel.lo[d]);
  }
  CEM_CUDA(cudaMemcpyAsync(h->mean_d, mean.data(), sizeof(float) * D, cudaMemcpyHostToDevice, h->stream));
  CEM_CUDA(cudaMemcpyAsync(h->chol_d, chol.data(), sizeof(float) * D * D, cudaMemcpyHostToDevice, h->stream));
  cudaError_t e = launch_sample(h->mean_d, h->chol_d, 12345, nullptr, 0, 0, N, D, h->theta_d, h->stream);
  if (e != cudaSuccess) return cuda_fail(e, "autotune sample");
  // candidates: threads per CTA (those that keep the CTAs within what the
  // SMs hold at once), and for pick-and-place also 8 or 32 lanes per
  // rollout; a lane width whose first shape is over twice the best so far
  // is dropped
  const int blocks1[] = {2, 4, 8, 16, 32, 64, 128, 256};
  const int blocksG[] = {32, 64, 128, 256};
  float best_ms = INFINITY;
  int best_b = 128, best_t = 1;
  for (int t : {1, 8, 32}) {
    if (t > 1 && !multi_lane) break;
    const int* bl = t == 1 ? blocks1 : blocksG;
    const int nb = t == 1 ? 8 : 4;
    for (int i = 0; i < nb; ++i) {
      const int b = bl[i];
      if (t == 1 && b < 16 && (long long)(N + b - 1) / b > 32LL * sms) continue;  // more CTAs than resident
      float tot = 0.0f;
      for (int rep = 0; rep < 3; ++rep) {
        CEM_CUDA(cudaEventRecord(h->ev0, h->stream));
        e = launch_rollout(h->scene_d, h->host.kind, h->theta_d, N, h->J_d, h->cls_d, b, t, nullptr, h->stream,
                           h->host.base_ctrl != 0);
        if (e != cudaSuccess) return cuda_fail(e, "autotune rollout");
        CEM_CUDA(cudaEventRecord(h->ev1, h->stream));
        CEM_CUDA(cudaEventSynchronize(h->ev1));
        float ms = 0.0f;
        CEM_CUDA(cudaEventElapsedTime(&ms, h->ev0, h->ev1));
        if (rep > 0) tot += ms;  // the first launch is a warm-up
      }
      if (tot < best_ms) {
        best_ms = tot;
        best_b = b;
        best_t = t;
      } else if (i == 0 && t > 1 && tot > 2.0f * best_ms) {
        break;
      }
    }
  }
  h->block = best_b;
  h->tpr = best_t;
  if (block_out) *block_out = best_b;
  if (h->graph) {  // the captured rollout used the old launch shape
    cudaGraphExecDestroy(h->graph);
    h->graph = nullptr;
  }
  if (cache_path) {
    std::ofstream o(cache_path, std::ios::app);
    o << key << "|" << best_b << "|" << best_t << "\n";
  }
  return CEM_OK;
}

}  // extern "C"
