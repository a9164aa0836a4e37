// Mapping operators and the fine-mesh outputs of a CGP step.
//
//   restrict_rhs : injection u_c = u_f[0, n_c) (Eq. 19) fused with the weak
//                  Poisson right-hand side b = Gx F_x + Gy F_y (Eqs. 12, 15).
//   prolong      : Eq. 20 on the 4-way split: coarse nodes copy, edge
//                  midpoints average their two end values.
//   lorentz      : per fine triangle grad(phi), j = sigma(-grad phi + u x B)
//                  (Eqs. 4, 7) and f = j x B (Eqs. 2, 8, 13-14), one thread per
//                  coarse triangle producing its four children.
#include "cgp_internal.h"

namespace cgp {
namespace {

// One thread per coarse row.  F is formed from the fine velocity at the
// coarse nodes (the prefix of the fine numbering), so no restricted copy is
// needed; it is written only when the caller asks for it.
//
// Latency of dependent loads (row, columns, velocity) bounds it, so a row's
// entries are taken eight at a time with their loads issued together, and the
// uniform factor (B_z or rho / dt) is applied to the row's sums instead of to
// every entry: two FP64 operations per entry instead of four.
// 512x256, one call: 13.4 -> 11.4 us, launch included.
template <int KIND>
__global__ void restrict_rhs_kernel(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                                    const double* __restrict__ Gx, const double* __restrict__ Gy,
                                    double factor, const double* __restrict__ u_f,
                                    const double* __restrict__ v_f, double* __restrict__ u_c,
                                    double* __restrict__ v_c, double* __restrict__ b) {
  constexpr int B = 8;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  // potential: F = (v B_z, -u B_z), the in-plane part of u x B with u_z = 0; pressure: F = (rho / dt) (u~, v~)
  const double* __restrict__ fx = KIND == CGP_RHS_POTENTIAL ? v_f : u_f;
  const double* __restrict__ fy = KIND == CGP_RHS_POTENTIAL ? u_f : v_f;
  const int k0 = rowptr[i], k1 = rowptr[i + 1];
  double sx = 0.0, sy = 0.0;
  for (int k = k0; k < k1; k += B) {
    int j[B];
    double gx[B], gy[B], x[B], y[B];
#pragma unroll
    for (int q = 0; q < B; ++q) j[q] = k + q < k1 ? col[k + q] : i;
#pragma unroll
    for (int q = 0; q < B; ++q) {
      gx[q] = k + q < k1 ? Gx[k + q] : 0.0;
      gy[q] = k + q < k1 ? Gy[k + q] : 0.0;
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
      x[q] = fx[j[q]];
      y[q] = fy[j[q]];
    }
#pragma unroll
    for (int q = 0; q < B; ++q) {
      if (k + q < k1) {
        sx = fma(gx[q], x[q], sx);
        sy = fma(gy[q], y[q], sy);
      }
    }
  }
  b[i] = factor * (KIND == CGP_RHS_POTENTIAL ? sx - sy : sx + sy);
  if (u_c) u_c[i] = u_f[i];
  if (v_c) v_c[i] = v_f[i];
}

// One level-1 node per thread: the coarse prefix copied, then the midpoints of the coarse edges.
__global__ void prolong_kernel(int n_c, int n_f, const int2* __restrict__ edges,
                               const double* __restrict__ xc, double* __restrict__ xf) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_f) return;
  if (i < n_c) {
    xf[i] = xc[i];
  } else {
    const int2 e = edges[i - n_c];
    xf[i] = (xc[e.x] + xc[e.y]) * 0.5;
  }
}

// One further level (Eq. 20 from level l to l + 1, in place): node n_l + e
// is the midpoint of level-l edge e, where the parent's shape functions are
// (1/2, 1/2, 0); level l's nodes are the prefix and already hold their values.
__global__ void prolong_level_kernel(int n_l, int e_l, const int2* __restrict__ edges, double* __restrict__ xf) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= e_l) return;
  const int2 ed = edges[e];
  xf[n_l + e] = (xf[ed.x] + xf[ed.y]) * 0.5;
}

// Ohm's law and the force with uniform B, u_z = 0 and the vertex means
// (u_b, v_b) = (su, sv) / 3:  j = sigma (u x B - grad phi) and j x B expand to
//   f_x = -su k1 + sv k2 - g_y k3,   f_y = su k2 - sv k4 + g_x k3,
// k1 = sigma (B_y^2 + B_z^2) / 3, k2 = sigma B_x B_y / 3, k3 = sigma B_z,
// k4 = sigma (B_x^2 + B_z^2) / 3, folded once on the host.
struct ForceCoef {
  double k1, k2, k3, k4;
};

// One thread per parent triangle and its four fine children.  A child of the
// midpoint split is the parent scaled by 1/2 (the middle child also turned by
// half a turn), so with the parent's b_i = y_j - y_k, c_i = x_k - x_j and doubled
// area a2 every child has grad phi = 2 sum_i phi_i (b_i, c_i) / a2.  The rows sum
// to zero, so two differences of phi and the parent's (b_1, b_2, c_1, c_2) 2 / a2,
// kept per parent since assembly (parent_shape_kernel), give a gradient in four
// operations, and the middle child's differences are two of the others'.
//
// The FP64 pipe bounds it (16 clocks a warp operation and SM): 20 operations a
// parent for the gradients and 38 for the force, against 50 and 38 when each
// launch formed the geometry and a division.  512x256 (262,144 parents): 48.4 -> 34.3 us
// with the force, 29.5 -> 15.0 us without (25 and 10 us of FP64 pipe).
template <bool FORCE>
__global__ void lorentz_kernel(int t_c, int t_f, const int* __restrict__ tri,
                               const int* __restrict__ mid, const double2* __restrict__ shape,
                               const double* __restrict__ phi, const double* __restrict__ u,
                               const double* __restrict__ v, ForceCoef k, double* __restrict__ grad,
                               double* __restrict__ force) {
  const int T = blockIdx.x * blockDim.x + threadIdx.x;
  if (T >= t_c) return;
  const int ia = tri[3 * T], ib = tri[3 * T + 1], ic = tri[3 * T + 2];
  const int iab = mid[3 * T], ibc = mid[3 * T + 1], ica = mid[3 * T + 2];
  const double2 b = shape[2 * (size_t)T], c = shape[2 * (size_t)T + 1];   // (b_1, b_2), (c_1, c_2), each 2 / a2
  const double pa = phi[ia], pb = phi[ib], pc = phi[ic], pab = phi[iab], pbc = phi[ibc], pca = phi[ica];
  // vertex sums of u and v for the four children, sharing the midpoint pairs
  double su[4] = {0, 0, 0, 0}, sv[4] = {0, 0, 0, 0};
  if (FORCE) {
    const double uab = u[iab], ubc = u[ibc], uca = u[ica], vab = v[iab], vbc = v[ibc], vca = v[ica];
    const double u_a = uab + uca, u_b = uab + ubc, u_c = uca + ubc;
    const double v_a = vab + vca, v_b = vab + vbc, v_c = vca + vbc;
    su[0] = u[ia] + u_a; su[1] = u[ib] + u_b; su[2] = u[ic] + u_c; su[3] = u_a + ubc;
    sv[0] = v[ia] + v_a; sv[1] = v[ib] + v_b; sv[2] = v[ic] + v_c; sv[3] = v_a + vbc;
  }
  // children (a, ab, ca), (ab, b, bc), (ca, bc, c): second and third vertex less the first; middle (ab, bc, ca)
  const double ba = pbc - pab, bc = pbc - pca;
  const double d1[4] = {pab - pa, pb - pab, bc, bc};
  const double d2[4] = {pca - pa, ba, pc - pca, ba};
  double gx[4], gy[4], fx[4], fy[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    gx[q] = fma(d2[q], b.y, d1[q] * b.x);
    gy[q] = fma(d2[q], c.y, d1[q] * c.x);
    if (FORCE) {
      fx[q] = sv[q] * k.k2 - su[q] * k.k1 - gy[q] * k.k3;
      fy[q] = su[q] * k.k2 - sv[q] * k.k4 + gx[q] * k.k3;
    }
  }
  const size_t t0 = 4 * (size_t)T;
  // four consecutive children: 32-byte aligned vector stores
  reinterpret_cast<double4*>(grad + t0)[0] = make_double4(gx[0], gx[1], gx[2], gx[3]);
  reinterpret_cast<double4*>(grad + t_f + t0)[0] = make_double4(gy[0], gy[1], gy[2], gy[3]);
  if (FORCE) {
    reinterpret_cast<double4*>(force + t0)[0] = make_double4(fx[0], fx[1], fx[2], fx[3]);
    reinterpret_cast<double4*>(force + t_f + t0)[0] = make_double4(fy[0], fy[1], fy[2], fy[3]);
  }
}

// (b_1, b_2) 2 / a2 and (c_1, c_2) 2 / a2 of every parent triangle.
__global__ void parent_shape_kernel(int t, const int* __restrict__ tri, const double2* __restrict__ xy,
                                    double2* __restrict__ shape) {
  const int T = blockIdx.x * blockDim.x + threadIdx.x;
  if (T >= t) return;
  const double2 xa = xy[tri[3 * T]], xb = xy[tri[3 * T + 1]], xc = xy[tri[3 * T + 2]];
  const double a2 = (xb.x - xa.x) * (xc.y - xa.y) - (xc.x - xa.x) * (xb.y - xa.y);
  const double inv2 = 2.0 / a2;
  shape[2 * (size_t)T] = make_double2((xc.y - xa.y) * inv2, (xa.y - xb.y) * inv2);
  shape[2 * (size_t)T + 1] = make_double2((xa.x - xc.x) * inv2, (xb.x - xa.x) * inv2);
}

// Velocity correction (Eqs. 16-17) at fine node i with the lumped P1 mass:
// u_i = u~_i - (dt/rho) sum_T |T| dp/dx|_T / sum_T |T| over the fine
// triangles T around i.  For T = (i, j, k) counter-clockwise,
// 2|T| grad p = (p_i (y_j - y_k) + p_j (y_k - y_i) + p_k (y_i - y_j),
//                p_i (x_k - x_j) + p_j (x_i - x_k) + p_k (x_j - x_i)).
// The right-hand side is linear in p with coefficients of the mesh alone, so the
// sums over the triangles are done once per mesh: row i of the operator holds
// the node itself and its neighbours with (w_x, w_y) of the mean gradient.
//
// Rows are stored in slices of 32 (one warp), entry q of the slice's rows side
// by side, so that every load of a warp is one contiguous 128 or 512 bytes;
// rows shorter than the slice's longest are filled with the node itself and
// zero weights.  14 FP64 operations a node instead of about 120, for 20 bytes an
// entry from memory: bound by both alike.  525,312
// nodes: 126 -> 21 us (97 MB).
__global__ void velocity_correct_kernel(int n_f, const long long* __restrict__ off, const int* __restrict__ col,
                                        const double2* __restrict__ coef, const double* __restrict__ p,
                                        const double* ut, const double* vt, double c, double* u, double* v) {
  constexpr int B = 7;   // an interior node of a triangular mesh has itself and about six neighbours
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_f) return;
  const long long e0 = off[i >> 5] + (i & 31), e1 = off[(i >> 5) + 1];
  const double u0 = ut[i], v0 = vt[i];
  double sx = 0.0, sy = 0.0;
  for (long long e = e0; e < e1; e += 32 * B) {
    int j[B];
    double2 w[B];
    double pj[B];
#pragma unroll
    for (int q = 0; q < B; ++q) j[q] = e + 32 * q < e1 ? col[e + 32 * q] : i;
#pragma unroll
    for (int q = 0; q < B; ++q) w[q] = e + 32 * q < e1 ? coef[e + 32 * q] : make_double2(0.0, 0.0);
#pragma unroll
    for (int q = 0; q < B; ++q) pj[q] = p[j[q]];
#pragma unroll
    for (int q = 0; q < B; ++q) {
      sx = fma(w[q].x, pj[q], sx);
      sy = fma(w[q].y, pj[q], sy);
    }
  }
  u[i] = fma(-c, sx, u0);
  v[i] = fma(-c, sy, v0);
}

// The operator's rows from the incidence lists (node i's triangles (i, j, k) as
// pairs (j, k)).  Entries of a row: the node, then its neighbours in the order
// of their first appearance.  Finding repeated neighbours compares every pair of
// a list; a list longer than kMergeEntries (a hub of more than 32 triangles)
// keeps an entry for each appearance instead, so that one thread's work on it
// stays linear (2000 triangles around a node, first call: 1.8 s compared, 1.6 ms
// before there was an operator).
constexpr int kMergeEntries = 64;
__device__ __forceinline__ bool first_seen(const int* __restrict__ ent, int e0, int e) {
  for (int f = e0; f < e; ++f)
    if (ent[f] == ent[e]) return false;
  return true;
}
__global__ void correct_count_kernel(int n_f, const int* __restrict__ ptr, const int* __restrict__ ent,
                                     int* __restrict__ width) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  int len = 0;
  if (i < n_f) {
    const int e0 = 2 * ptr[i], e1 = 2 * ptr[i + 1];
    len = 1;
    if (e1 - e0 > kMergeEntries) len += e1 - e0;
    else
      for (int e = e0; e < e1; ++e) len += first_seen(ent, e0, e) ? 1 : 0;
  }
  const int most = __reduce_max_sync(0xffffffffu, len);
  if ((i & 31) == 0 && i < n_f) width[i >> 5] = most;
}
__global__ void correct_fill_kernel(int n_f, const int* __restrict__ ptr, const int* __restrict__ ent,
                                    const double2* __restrict__ xy, const long long* __restrict__ off,
                                    int* __restrict__ col, double2* __restrict__ coef) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_f) return;
  const int e0 = 2 * ptr[i], e1 = 2 * ptr[i + 1];
  const double2 xi = xy[i];
  double sa = 0.0, ox = 0.0, oy = 0.0;
  for (int e = e0; e < e1; e += 2) {
    const double2 xj = xy[ent[e]], xk = xy[ent[e + 1]];
    ox += xj.y - xk.y;
    oy += xk.x - xj.x;
    sa += (xj.x - xi.x) * (xk.y - xi.y) - (xk.x - xi.x) * (xj.y - xi.y);
  }
  const double ia = 1.0 / sa;
  long long at = off[i >> 5] + (i & 31);
  const long long end = off[(i >> 5) + 1];
  col[at] = i;
  coef[at] = make_double2(ox * ia, oy * ia);
  at += 32;
  if (e1 - e0 > kMergeEntries) {
#pragma unroll 8
    for (int e = e0; e < e1; e += 2) {   // a hub, triangle by triangle: independent loads in flight
      const int j = ent[e], k = ent[e + 1];
      const double2 xj = xy[j], xk = xy[k];
      const long long q = at + 32LL * (e - e0);
      col[q] = j;
      coef[q] = make_double2((xk.y - xi.y) * ia, (xi.x - xk.x) * ia);
      col[q + 32] = k;
      coef[q + 32] = make_double2((xi.y - xj.y) * ia, (xj.x - xi.x) * ia);
    }
    at += 32LL * (e1 - e0);
  } else {
    for (int e = e0; e < e1; ++e) {
      if (!first_seen(ent, e0, e)) continue;
      double wx = 0.0, wy = 0.0;
      for (int f = e0; f < e1; ++f) {
        if (ent[f] != ent[e]) continue;
        const bool second = (f - e0) & 1;   // this neighbour is k of (i, j, k), else j
        const double2 xo = xy[ent[second ? f - 1 : f + 1]];
        wx += second ? xi.y - xo.y : xo.y - xi.y;
        wy += second ? xo.x - xi.x : xi.x - xo.x;
      }
      col[at] = ent[e];
      coef[at] = make_double2(wx * ia, wy * ia);
      at += 32;
    }
  }
  for (; at < end; at += 32) {
    col[at] = i;
    coef[at] = make_double2(0.0, 0.0);
  }
}

}  // namespace

int launch_restrict_rhs(cgp_mesh_impl* m, int kind, double bz, double rho_over_dt, const double* u_f,
                        const double* v_f, double* u_c, double* v_c, double* b, cudaStream_t s) {
  const int bs = 128, gs = (m->n_c + bs - 1) / bs;
  if (kind == CGP_RHS_POTENTIAL)
    restrict_rhs_kernel<CGP_RHS_POTENTIAL><<<gs, bs, 0, s>>>(m->n_c, m->rowptr, m->col, m->Gx, m->Gy, bz,
                                                             u_f, v_f, u_c, v_c, b);
  else
    restrict_rhs_kernel<CGP_RHS_PRESSURE><<<gs, bs, 0, s>>>(m->n_c, m->rowptr, m->col, m->Gx, m->Gy, rho_over_dt,
                                                            u_f, v_f, u_c, v_c, b);
  CGP_CUDA(cudaGetLastError());
  return CGP_OK;
}

int launch_prolong(cgp_mesh_impl* m, const double* xc, double* xf, cudaStream_t s) {
  const int bs = 256;
  const int n1 = m->h_lvl_nodes[1];
  prolong_kernel<<<(n1 + bs - 1) / bs, bs, 0, s>>>(m->n_c, n1, reinterpret_cast<const int2*>(m->edges), xc, xf);
  CGP_CUDA(cudaGetLastError());
  for (int l = 1; l < m->levels; ++l) {   // one launch per further level, as Eq. 20 prolongs one level at a time
    const int e_l = m->h_lvl_eoff[l + 1] - m->h_lvl_eoff[l];
    prolong_level_kernel<<<(e_l + bs - 1) / bs, bs, 0, s>>>(
        m->h_lvl_nodes[l], e_l, reinterpret_cast<const int2*>(m->edges) + m->h_lvl_eoff[l], xf);
    CGP_CUDA(cudaGetLastError());
  }
  return CGP_OK;
}

int launch_lorentz(cgp_mesh_impl* m, const double* phi, const double* u, const double* v, const double B[3],
                   double sigma, double* grad, double* force, cudaStream_t s) {
  // one thread per parent (level levels - 1) triangle and its four fine children
  const int bs = 128, gs = (m->t_par + bs - 1) / bs;
  const double2* shape = reinterpret_cast<const double2*>(m->shape_par);
  const ForceCoef k{sigma * (B[1] * B[1] + B[2] * B[2]) / 3.0, sigma * B[0] * B[1] / 3.0, sigma * B[2],
                    sigma * (B[0] * B[0] + B[2] * B[2]) / 3.0};
  if (force)
    lorentz_kernel<true><<<gs, bs, 0, s>>>(m->t_par, m->t_f, m->tri_par, m->mid_par, shape, phi, u, v, k, grad, force);
  else
    lorentz_kernel<false><<<gs, bs, 0, s>>>(m->t_par, m->t_f, m->tri_par, m->mid_par, shape, phi, u, v, k, grad, force);
  CGP_CUDA(cudaGetLastError());
  return CGP_OK;
}

int launch_parent_shape(cgp_mesh_impl* m, cudaStream_t s) {
  parent_shape_kernel<<<(m->t_par + 255) / 256, 256, 0, s>>>(m->t_par, m->tri_par,
                                                             reinterpret_cast<const double2*>(m->xy_f),
                                                             reinterpret_cast<double2*>(m->shape_par));
  CGP_CUDA(cudaGetLastError());
  return CGP_OK;
}

// The velocity correction's operator, built once per mesh: the incidence lists
// on the host, the rows on the GPU.  The map calls share no scratch, so several
// host threads may make them on one mesh: one of them builds, the others wait.
static int build_correction(cgp_mesh_impl* m, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(m->vop_mu);
  if (m->vop_base) return CGP_OK;
  const std::vector<int>& tp = m->levels >= 2 ? m->h_tri_par : m->h_tri_c;
  const std::vector<int>& mp = m->levels >= 2 ? m->h_mid_par : m->h_tri_mid;
  const size_t nf = m->n_f, tf = m->t_f;
  std::vector<int> ptr(nf + 1, 0), ent(6 * tf);
  auto fine_tri = [&](size_t t, int (&v)[3]) {
    const size_t T = t / 4;
    const int a = tp[3 * T], b = tp[3 * T + 1], c = tp[3 * T + 2];
    const int mab = mp[3 * T], mbc = mp[3 * T + 1], mca = mp[3 * T + 2];
    const int ch[4][3] = {{a, mab, mca}, {mab, b, mbc}, {mca, mbc, c}, {mab, mbc, mca}};
    for (int l = 0; l < 3; ++l) v[l] = ch[t % 4][l];
  };
  int v[3];
  for (size_t t = 0; t < tf; ++t) {
    fine_tri(t, v);
    for (int l = 0; l < 3; ++l) ptr[v[l] + 1]++;
  }
  for (size_t i = 0; i < nf; ++i) ptr[i + 1] += ptr[i];
  std::vector<int> fill(ptr.begin(), ptr.end() - 1);
  for (size_t t = 0; t < tf; ++t) {
    fine_tri(t, v);
    for (int l = 0; l < 3; ++l) {
      const int q = fill[v[l]]++;
      ent[2 * (size_t)q] = v[(l + 1) % 3];
      ent[2 * (size_t)q + 1] = v[(l + 2) % 3];
    }
  }
  auto al = [](size_t v) { return (v + 255) / 256 * 256; };
  const size_t ns = (nf + 31) / 32;   // slices
  const size_t o_ent = al((nf + 1) * 4), o_width = o_ent + al(ent.size() * 4);
  char* lists = nullptr;
  CGP_CUDA(cudaMalloc(&lists, o_width + ns * 4));
  std::vector<int> width(ns);
  std::vector<long long> off(ns + 1, 0);
  char* base = nullptr;
  size_t o_col = 0, o_coef = 0;
  const int bs = 128, gs = (int)((nf + bs - 1) / bs);
  auto run = [&]() -> cudaError_t {
    cudaError_t e = cudaMemcpyAsync(lists, ptr.data(), (nf + 1) * 4, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaMemcpyAsync(lists + o_ent, ent.data(), ent.size() * 4, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) return e;
    correct_count_kernel<<<gs, bs, 0, s>>>((int)nf, (const int*)lists, (const int*)(lists + o_ent), (int*)(lists + o_width));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(width.data(), lists + o_width, ns * 4, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    for (size_t q = 0; q < ns; ++q) off[q + 1] = off[q] + 32LL * width[q];
    o_col = al((ns + 1) * 8);
    o_coef = o_col + al((size_t)off[ns] * 4);
    if ((e = cudaMalloc(&base, o_coef + (size_t)off[ns] * 16)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(base, off.data(), (ns + 1) * 8, cudaMemcpyHostToDevice, s)) != cudaSuccess) return e;
    correct_fill_kernel<<<gs, bs, 0, s>>>((int)nf, (const int*)lists, (const int*)(lists + o_ent),
                                          reinterpret_cast<const double2*>(m->xy_f), (const long long*)base,
                                          (int*)(base + o_col), (double2*)(base + o_coef));
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return cudaStreamSynchronize(s);
  };
  const cudaError_t e = run();
  cudaFree(lists);
  if (e != cudaSuccess) {
    cudaFree(base);
    return cuda_fail(e, "velocity correction operator");
  }
  m->vop_base = base;
  m->vop_off = (long long*)base;
  m->vop_col = (int*)(base + o_col);
  m->vop_coef = (double*)(base + o_coef);
  return CGP_OK;
}

int launch_velocity_correct(cgp_mesh_impl* m, const double* p_f, const double* u_t, const double* v_t,
                            double dt_over_rho, double* u, double* v, cudaStream_t s) {
  int st = build_correction(m, s);
  if (st != CGP_OK) return st;
  const int bs = 128;
  velocity_correct_kernel<<<(m->n_f + bs - 1) / bs, bs, 0, s>>>(
      m->n_f, m->vop_off, m->vop_col, reinterpret_cast<const double2*>(m->vop_coef), p_f, u_t, v_t, dt_over_rho, u, v);
  CGP_CUDA(cudaGetLastError());
  return CGP_OK;
}

}  // namespace cgp

using namespace cgp;

extern "C" int cgp_velocity_correct(cgp_mesh m, const double* p_f, const double* u_t, const double* v_t,
                                    double dt_over_rho, double* u, double* v, void* stream) {
  if (!m) return fail(CGP_ERR_INVALID_ARG, "cgp_velocity_correct: NULL mesh");
  if (!p_f || !u_t || !v_t || !u || !v) return fail(CGP_ERR_INVALID_ARG, "cgp_velocity_correct: NULL vector");
  if (!(dt_over_rho == dt_over_rho)) return fail(CGP_ERR_INVALID_ARG, "cgp_velocity_correct: dt_over_rho is NaN");
  return launch_velocity_correct(m, p_f, u_t, v_t, dt_over_rho, u, v, (cudaStream_t)stream);
}

static bool aligned(const void* p, size_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

extern "C" int cgp_restrict(cgp_mesh m, int kind, const double* B, double rho_over_dt, const double* u_f,
                            const double* v_f, double* u_c, double* v_c, double* b, void* stream) {
  if (!m) return fail(CGP_ERR_INVALID_ARG, "cgp_restrict: NULL mesh");
  if (!u_f || !v_f || !b) return fail(CGP_ERR_INVALID_ARG, "cgp_restrict: NULL u_f, v_f or b");
  if (kind != CGP_RHS_POTENTIAL && kind != CGP_RHS_PRESSURE)
    return fail(CGP_ERR_INVALID_ARG, "cgp_restrict: unknown kind");
  if (kind == CGP_RHS_POTENTIAL && !B) return fail(CGP_ERR_INVALID_ARG, "cgp_restrict: NULL B");
  const double bz = B ? B[2] : 0.0;
  return launch_restrict_rhs(m, kind, bz, rho_over_dt, u_f, v_f, u_c, v_c, b, (cudaStream_t)stream);
}

extern "C" int cgp_prolong(cgp_mesh m, const double* x_c, double* x_f, void* stream) {
  if (!m) return fail(CGP_ERR_INVALID_ARG, "cgp_prolong: NULL mesh");
  if (!x_c || !x_f) return fail(CGP_ERR_INVALID_ARG, "cgp_prolong: NULL vector");
  return launch_prolong(m, x_c, x_f, (cudaStream_t)stream);
}

extern "C" int cgp_lorentz(cgp_mesh m, const double* phi_f, const double* u_f, const double* v_f,
                           const double* B, double sigma, double* grad, double* force, void* stream) {
  if (!m) return fail(CGP_ERR_INVALID_ARG, "cgp_lorentz: NULL mesh");
  if (!phi_f || !grad || !B) return fail(CGP_ERR_INVALID_ARG, "cgp_lorentz: NULL phi_f, grad or B");
  if (force && (!u_f || !v_f)) return fail(CGP_ERR_INVALID_ARG, "cgp_lorentz: force needs u_f and v_f");
  if (!aligned(grad, 32) || (force && !aligned(force, 32)))
    return fail(CGP_ERR_INVALID_ARG, "cgp_lorentz: grad and force must be 32-byte aligned");
  // without force the velocity is not read; pass phi as a valid stand-in pointer
  const double* u = u_f ? u_f : phi_f;
  const double* v = v_f ? v_f : phi_f;
  return launch_lorentz(m, phi_f, u, v, B, sigma, grad, force, (cudaStream_t)stream);
}
