// Red/black SOR for the control variates' Poisson solves (sor.cuh).
//
// One kernel per half-sweep over all boxes.  In FP64 an update costs 5
// additions and 2 fma (omega / 6 is folded into the density, so there is no
// division), and GB300's FP64 rate, 16 cycles per warp instruction and SM,
// makes 128^3 take 11.7 us per half-sweep whatever else is done; the layout
// (split colours, zero ghosts, no bounds checks) leaves little else to wait
// for: neighbouring threads read neighbouring elements, every load of a
// thread's site is issued before the first addition.  The launches depend on
// one another programmatically, so that a launch's start (4 us by itself, more
// than the work of a small box) overlaps the end of the one before.
// Measured, us per half-sweep, before (natural order, every second thread
// idle, 64-bit divisions for the coordinates, an FP64 division) -> now: 16^3
// 4.2 -> 1.5, 48 x 40 x 44 8.3 -> 2.6, 64^3 12.6 -> 4.3, 128^3 69.9 -> 14.9 (18.4
// without the programmatic launches); 256 boxes of 32^3 .. 96^3, 626
// iterations, 3.42 -> 0.70 s.  Two sites per thread: 96^3 9.6 instead of 7.3,
// the same at 128^3; 256 threads: 48 x 40 x 44 4.7 instead of 2.8.
#include <algorithm>
#include <cmath>

#include "sor.cuh"

namespace coulps {
namespace {

constexpr int kSorThreads = 128;

struct SorItem {
  int box, z;
  int first;  // first of the item's sites of plane z, numbered y Wh + h
};

__global__ void __launch_bounds__(kSorThreads)
    sor_kernel(double *__restrict__ u, const double *__restrict__ r,
               const SorBox *__restrict__ boxes, const SorItem *__restrict__ items, int colour) {
  asm volatile("griddepcontrol.launch_dependents;");
  const SorItem it = items[blockIdx.x];
  const SorBox b = boxes[it.box];
  const long long plane = (long long)(b.Ly + 2) * b.Ws;
  const int t = it.first + (int)threadIdx.x;
  const int y = t / b.Wh, h = t - y * b.Wh;
  const int par = (colour + y + it.z) & 1;
  if (t >= b.Ly * b.Wh || 2 * h + par >= b.Lx) return;  // (sor_solve: not every thread)
  const long long at = b.off + (long long)colour * b.colour + (it.z + 1) * plane +
                       (long long)(y + 1) * b.Ws + h;
  const double *o = u + at + (colour ? -b.colour : b.colour);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const double zm = o[-plane], zp = o[plane], ym = o[-b.Ws], yp = o[b.Ws], c = o[0],
               e = o[par ? 1 : -1], w = u[at], q = r[at];
  const double S = ((zm + zp) + (ym + yp)) + (c + e);
  u[at] = fma(b.a, w, fma(b.b, S, -q));
}

__global__ void sor_scatter_kernel(const SorCharge *__restrict__ c, int64_t n,
                                   double *__restrict__ r, double *__restrict__ rho_nat) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const SorCharge q = c[i];
  r[q.at] = q.bq;
  rho_nat[q.nat] = q.q;
}

__global__ void sor_natural_kernel(const double *__restrict__ u, const SorBox *__restrict__ boxes,
                                   const SorItem *__restrict__ items,
                                   double *__restrict__ u_nat) {
  const SorItem it = items[blockIdx.x];
  const SorBox b = boxes[it.box];
  const int n = b.Ly * b.Wh;
  const int t = it.first + (int)threadIdx.x;
  if (t >= n) return;
  const int y = t / b.Wh, h = t - y * b.Wh;
  const double *src = u + b.off + ((long long)(it.z + 1) * (b.Ly + 2) + y + 1) * b.Ws + h;
  double *dst = u_nat + b.nat + ((long long)it.z * b.Ly + y) * b.Lx + 2 * h;
  const int p = (y + it.z) & 1;  // colour of site 2 h
  dst[0] = src[p ? b.colour : 0];
  if (2 * h + 1 < b.Lx) dst[1] = src[p ? 0 : b.colour];
}

// The same update in the natural-order arrays (every second thread has no site).
__global__ void __launch_bounds__(kSorThreads)
    sor_in_place_kernel(double *__restrict__ u, const double *__restrict__ rho, const SorBox b,
                        int colour) {
  const long long n = (long long)b.Lx * b.Ly * b.Lz, row = b.Lx, plane = row * b.Ly;
  double *us = u + b.nat;
  for (long long i = (long long)blockIdx.x * kSorThreads + threadIdx.x; i < n;
       i += (long long)gridDim.x * kSorThreads) {
    const int z = (int)(i / plane), y = (int)(i / row - (long long)z * b.Ly),
              x = (int)(i - (i / row) * row);
    if (((x + y + z) & 1) != colour) continue;
    const double zm = z > 0 ? us[i - plane] : 0.0, zp = z + 1 < b.Lz ? us[i + plane] : 0.0;
    const double ym = y > 0 ? us[i - row] : 0.0, yp = y + 1 < b.Ly ? us[i + row] : 0.0;
    const double xm = x > 0 ? us[i - 1] : 0.0, xp = x + 1 < b.Lx ? us[i + 1] : 0.0;
    const double S = ((zm + zp) + (ym + yp)) + (xm + xp);
    us[i] = fma(b.a, us[i], fma(b.b, S, -__dmul_rn(b.b, rho[b.nat + i])));
  }
}

// Where the split arrays do not fit in device memory: the solve in u_nat and
// rho_nat alone, box by box, with no allocation.  Bitwise the same u; 400
// iterations of 64^3 / 128^3 with the set-up around them 6.8 / 30.2 ms instead of
// 4.0 / 12.7.
cudaError_t solve_in_place(const std::vector<SorBox> &boxes, const std::vector<SorCharge> &charges,
                           int n_iter, size_t nat, double *u_nat, double *rho_nat,
                           cudaStream_t s) {
  std::vector<double> rho(nat, 0.0);
  for (const SorCharge &c : charges) rho[c.nat] = c.q;
  cudaError_t e = cudaMemsetAsync(u_nat, 0, nat * sizeof(double), s);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(rho_nat, rho.data(), nat * sizeof(double), cudaMemcpyHostToDevice, s);
  for (const SorBox &b : boxes) {
    const long long n = (long long)b.Lx * b.Ly * b.Lz;
    const unsigned grid = (unsigned)std::min<long long>((n + kSorThreads - 1) / kSorThreads, 8192);
    for (int i = 0; i < 2 * n_iter && e == cudaSuccess; ++i) {
      sor_in_place_kernel<<<grid, kSorThreads, 0, s>>>(u_nat, rho_nat, b, i & 1);
      e = cudaGetLastError();
    }
  }
  const cudaError_t es = cudaStreamSynchronize(s);  // the host density leaves scope
  return e == cudaSuccess ? es : e;
}

}  // namespace

SorBox sor_box(int Lx, int Ly, int Lz, long long off, long long nat) {
  SorBox b;
  b.Lx = Lx;
  b.Ly = Ly;
  b.Lz = Lz;
  b.Wh = (Lx + 1) / 2;
  b.Ws = b.Wh + 1;
  b.off = off;
  b.nat = nat;
  b.colour = (long long)(Lz + 2) * (Ly + 2) * b.Ws;
  // SOR factor from the Jacobi spectral radius of the Dirichlet box
  const double rj = (std::cos(M_PI / (Lx + 1)) + std::cos(M_PI / (Ly + 1)) +
                     std::cos(M_PI / (Lz + 1))) / 3.0;
  const double omega = 2.0 / (1.0 + std::sqrt(1.0 - rj * rj));
  b.a = 1.0 - omega;
  b.b = omega / 6.0;
  return b;
}

void sor_charges(const SorBox &b, int64_t n, const int32_t *sites, const double *q,
                 std::vector<SorCharge> &out) {
  const size_t first = out.size();
  for (int64_t i = 0; i < n; ++i) {
    const int32_t *p = sites + 3 * i;
    SorCharge c;
    c.at = b.off + (long long)((p[0] + p[1] + p[2]) & 1) * b.colour +
           ((long long)(p[2] + 1) * (b.Ly + 2) + p[1] + 1) * b.Ws + (p[0] >> 1);
    c.nat = b.nat + ((long long)p[2] * b.Ly + p[1]) * b.Lx + p[0];
    c.q = q[i];
    c.bq = 0.0;
    out.push_back(c);
  }
  std::stable_sort(out.begin() + first, out.end(),
                   [](const SorCharge &x, const SorCharge &y) { return x.nat < y.nat; });
  size_t m = first;
  for (size_t i = first; i < out.size(); ++i) {
    if (m > first && out[m - 1].nat == out[i].nat)
      out[m - 1].q += out[i].q;
    else
      out[m++] = out[i];
  }
  out.resize(m);
  for (size_t i = first; i < m; ++i) out[i].bq = b.b * out[i].q;
}

cudaError_t sor_solve(const std::vector<SorBox> &boxes, const std::vector<SorCharge> &charges,
                      int n_iter, double *u_nat, double *rho_nat, const Allocator &alloc,
                      cudaStream_t s) {
  long long elems = 0, nat = 0;
  for (const SorBox &b : boxes) {
    elems += sor_elems(b);
    nat += (long long)b.Lx * b.Ly * b.Lz;
  }
  std::vector<SorItem> items;
  for (size_t k = 0; k < boxes.size(); ++k) {
    const int n = boxes[k].Ly * boxes[k].Wh;
    for (int z = 0; z < boxes[k].Lz; ++z)
      for (int t = 0; t < n; t += kSorThreads) items.push_back(SorItem{(int)k, z, t});
  }
  const size_t bytes_u = (size_t)elems * sizeof(double);
  double *u = (double *)dev_alloc(alloc, bytes_u, s), *r = (double *)dev_alloc(alloc, bytes_u, s);
  SorBox *d_boxes = (SorBox *)dev_alloc(alloc, boxes.size() * sizeof(SorBox), s);
  SorItem *d_items = (SorItem *)dev_alloc(alloc, items.size() * sizeof(SorItem), s);
  SorCharge *d_q = (SorCharge *)dev_alloc(alloc, charges.size() * sizeof(SorCharge), s);
  auto release = [&]() {
    for (void *p : {(void *)u, (void *)r, (void *)d_boxes, (void *)d_items, (void *)d_q})
      dev_free(alloc, p, s);
  };
  if (!u || !r || !d_boxes || !d_items || !d_q) {
    release();
    return solve_in_place(boxes, charges, n_iter, (size_t)nat, u_nat, rho_nat, s);
  }
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
    return e == cudaSuccess;
  };
  auto up = [&](void *d, const void *h, size_t n) {
    if (n > 0 && e == cudaSuccess) ok(cudaMemcpyAsync(d, h, n, cudaMemcpyHostToDevice, s));
  };
  up(d_boxes, boxes.data(), boxes.size() * sizeof(SorBox));
  up(d_items, items.data(), items.size() * sizeof(SorItem));
  up(d_q, charges.data(), charges.size() * sizeof(SorCharge));
  if (e == cudaSuccess) ok(cudaMemsetAsync(u, 0, bytes_u, s));
  if (e == cudaSuccess) ok(cudaMemsetAsync(r, 0, bytes_u, s));
  if (e == cudaSuccess) ok(cudaMemsetAsync(rho_nat, 0, (size_t)nat * sizeof(double), s));
  if (e == cudaSuccess && !charges.empty()) {
    sor_scatter_kernel<<<(unsigned)((charges.size() + 255) / 256), 256, 0, s>>>(
        d_q, (int64_t)charges.size(), r, rho_nat);
    ok(cudaGetLastError());
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)items.size());
  cfg.blockDim = dim3(kSorThreads);
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  // Threads without a site leave before their wait, so every launch needs one that
  // stays: a launch of which all threads had left would end before the launch ahead
  // of it, and the launch behind it would then run beside that one.  Colour 0 has a
  // site in every box, colour 1 in those of more than one; without any its launches
  // have nothing to do and are not made.  (One thread of every CTA waiting instead
  // costs 128^3 0.5%, every idle thread 48 x 40 x 44 5.0 instead of 2.6 us.)
  int colours = 1;
  for (const SorBox &b : boxes)
    if ((long long)b.Lx * b.Ly * b.Lz > 1) colours = 2;
  for (int i = 0; i < n_iter && e == cudaSuccess; ++i)
    for (int c = 0; c < colours && e == cudaSuccess; ++c)
      ok(cudaLaunchKernelEx(&cfg, sor_kernel, u, (const double *)r, (const SorBox *)d_boxes,
                            (const SorItem *)d_items, c));
  if (e == cudaSuccess) {
    sor_natural_kernel<<<(unsigned)items.size(), kSorThreads, 0, s>>>(u, d_boxes, d_items, u_nat);
    ok(cudaGetLastError());
  }
  // the host lists leave scope with this call
  const cudaError_t es = cudaStreamSynchronize(s);
  ok(es);
  release();
  return e;
}

}  // namespace coulps
