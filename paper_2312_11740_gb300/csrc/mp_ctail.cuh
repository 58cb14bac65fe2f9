// Coarse tail of the V-cycle on one thread-block cluster (A6-A9).
//
// Below some ten thousand cells every V-cycle kernel is latency-bound: a
// half-sweep of a 16^3 level is a launch of ~2 us whatever its size.  One launch of
// a cluster of up to CT_MAX_CTAS CTAs runs the top level it can take (32^3 at
// 256^3) and every coarser one: sweeps, restrictions, prolongations and the
// coarsest solve.
//
// Every level is cut in y and z (whole x rows, cuts at even y and z) into at
// most one block per CTA; a small level takes fewer blocks, down to one, whose
// half-sweeps need no exchange.  Between half-sweeps a CTA writes the new values of
// its boundary rows straight into the shared memory of the blocks beside it
// (distributed shared memory), each as a word that carries its half-sweep's epoch, and
// polls its own shared memory for theirs: no cluster barrier, which waits for
// the slowest CTA and costs ~0.8 us, inside a level.  Slots alternate with the epoch's
// parity, so a word is overwritten only after its reader has sent its own next
// message.  Cluster barriers separate levels.  Waits are bounded: a CTA that gives
// up sets *err and finishes without waiting (its result is not used).
//
// Shared-memory arrays are split by colour as in mp_visit.cuh; a level's strides
// come from its largest block, so a cell's address in its owner's shared memory
// follows from its indices.  The coarsest level is replicated in every CTA.
//
// Same algorithm and arithmetic per cell as k_tail: red-black Gauss-Seidel
// on the level's own faces with the stored 1/diag, colour 0 first on the way
// down and last on the way up (a symmetric preconditioner), difference-form
// residuals, restriction by half the sum of the 8 children, piecewise-constant
// prolongation, and the dense FP64 coarsest inverse.
#pragma once

#include <cooperative_groups.h>

namespace mp {

namespace cgx = cooperative_groups;

constexpr int CT_MAX_CTAS = 16, CTL_THREADS = 512, CT_MAX_LEVELS = 10, CT_MAX_COARSE = 512;
constexpr int CT_POLL = 1 << 22;  // polls of one wait (tenths of a second)

template <typename T>
struct CtLevel {
  Dims d;
  int n, nu1, nu2;
  int py, pz, bym, bzm;  // blocks, and the largest block's rows and planes
  int off;               // element offset of the level's arrays in shared memory
  const T *bx, *by, *bz, *idiag, *dd;  // level arrays (dd null without outflow)
};
template <typename T>
struct CtArgs {
  int nlev;  // levels of the tail (the last one is the coarsest)
  CtLevel<T> lv[CT_MAX_LEVELS];
  const double *Minv;
  int singular;   // mean-project the coarsest right-hand side
  int mail;       // byte offset of the exchange slots
  int mail_words;  // 8-byte words of both parities
  double *err;
};

// Elements of a level's arrays in one CTA: x with halo, b, 1/diag, faces,
// outflow diagonal.  Coarsest level: x and b.
__host__ __device__ inline int ct_elems(const Dims &d, int bym, int bzm, bool dd, bool coarsest) {
  if (coarsest) return 2 * d.nx * d.ny * d.nz;
  const int own = bym * bzm;
  return d.nx * ((bym + 2) * (bzm + 2) + 3 * own + (bym + 1) * bzm + bym * (bzm + 1) +
                 (dd ? own : 0));
}
__host__ __device__ inline int ct_slots(const Dims &d, int bym, int bzm) {
  return (bym + bzm) * d.nx;  // y-low, y-high (planes x pairs), z-low, z-high (rows x pairs)
}

__device__ __forceinline__ uint32_t ct_map(uint32_t addr, int rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void ct_st64(uint32_t addr, unsigned long long v) {
  asm volatile("st.relaxed.cluster.shared::cluster.u64 [%0], %1;" ::"r"(addr), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long ct_ld64(uint32_t addr) {
  unsigned long long v;
  asm volatile("ld.relaxed.cluster.shared::cta.u64 %0, [%1];" : "=l"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void ct_send(uint32_t addr, float v, unsigned e) {
  ct_st64(addr, ((unsigned long long)e << 32) | __float_as_uint(v));
}
__device__ __forceinline__ void ct_send(uint32_t addr, double v, unsigned e) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  ct_st64(addr, ((unsigned long long)e << 32) | (u & 0xffffffffull));
  ct_st64(addr + 8, ((unsigned long long)e << 32) | (u >> 32));
}
__device__ __forceinline__ bool ct_recv(uint32_t addr, unsigned e, float &v) {
  const unsigned long long w = ct_ld64(addr);
  v = __uint_as_float((unsigned)w);
  return (unsigned)(w >> 32) == e;
}
__device__ __forceinline__ bool ct_recv(uint32_t addr, unsigned e, double &v) {
  const unsigned long long a = ct_ld64(addr), b = ct_ld64(addr + 8);
  v = __longlong_as_double((long long)((a & 0xffffffffull) | (b << 32)));
  return (unsigned)(a >> 32) == e && (unsigned)(b >> 32) == e;
}
__device__ __forceinline__ void ct_st(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void ct_st(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ float ct_ld(uint32_t addr, float) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ double ct_ld(uint32_t addr, double) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr) : "memory");
  return v;
}
// (n / 2) units of two rows cut into p parts [c u / p, (c + 1) u / p): first row
// of part c, and the part that holds a row
__host__ __device__ inline int ct_cut(int n, int p, int c) { return 2 * (c * (n >> 1) / p); }
__host__ __device__ inline int ct_part(int n, int p, int row) {
  return (((row >> 1) + 1) * p - 1) / (n >> 1);
}

// One level seen by one CTA.
template <typename T>
struct CtView {
  T *X, *B, *ID, *HX, *HY, *HZ, *DD;
  int nx, ny, nz, P, py, pz, bym, bzm, cy, cz, y0, by, z0, bz;
  int n1, nh, n1y, n1z;
  bool own;  // this CTA holds a block
  __device__ CtView(T *base, const CtLevel<T> &l, int rank) {
    nx = l.d.nx, ny = l.d.ny, nz = l.d.nz, P = nx >> 1;
    py = l.py, pz = l.pz, bym = l.bym, bzm = l.bzm;
    own = rank < py * pz;
    cy = own ? rank % py : 0, cz = own ? rank / py : 0;
    y0 = ct_cut(ny, py, cy), by = ct_cut(ny, py, cy + 1) - y0;
    z0 = ct_cut(nz, pz, cz), bz = ct_cut(nz, pz, cz + 1) - z0;
    n1 = bym * bzm * P, nh = (bym + 2) * (bzm + 2) * P;
    n1y = (bym + 1) * bzm * P, n1z = bym * (bzm + 1) * P;
    X = base + l.off;
    B = X + 2 * nh;
    ID = B + 2 * n1;
    HX = ID + 2 * n1;
    HY = HX + 2 * n1;
    HZ = HY + 2 * n1y;
    DD = l.dd ? HZ + 2 * n1z : nullptr;
  }
  __device__ int f(int p, int ly, int lz) const { return (lz * bym + ly) * P + p; }
  __device__ int h(int p, int ly, int lz) const {
    return ((lz + 1) * (bym + 2) + ly + 1) * P + p;
  }
};

// The walk of a thread over its cells: one pair p, rows advancing by rpt.
struct CtWalk {
  int p, act, ly0, lz0, dly, dlz;
  bool works;
  __device__ CtWalk(int P, int by) {
    const int tid = threadIdx.x, rpt = CTL_THREADS / P;
    act = rpt * P;
    works = tid < act;
    const int r0 = tid / P;
    p = tid - r0 * P;
    lz0 = r0 / by, ly0 = r0 - lz0 * by;
    dlz = rpt / by, dly = rpt - dlz * by;
  }
};

// One colour of one sweep on this CTA's block, and the exchange of its boundary
// rows under epoch e (0: none).  zero: x is taken as zero.  mail: local address of the slots.
template <typename T, int C>
__device__ __forceinline__ void ct_half(const CtView<T> &v, const CtWalk &w, bool zero, unsigned e,
                                        uint32_t mail, const uint32_t rem[4], uint32_t flip,
                                        bool &dead, double *err) {
  constexpr int W = sizeof(T) == 8 ? 16 : 8;  // bytes of a slot
  const int P = v.P, by = v.by, bz = v.bz, sZ = (v.bym + 2) * P;
  const int dlo = w.p == 0 ? P - 1 : -1, dhi = w.p == P - 1 ? 1 - P : 1;
  const int par = v.y0 + v.z0 + C, ncta = v.py * v.pz;
  const bool exchange = e != 0u && ncta > 1;
  const uint32_t m = (e & 1u) ? flip : 0u;
  T *Xc = v.X + C * v.nh;
  const T *Xo = v.X + (1 - C) * v.nh;
  if (w.works) {
    int ly = w.ly0, lz = w.lz0;
    for (int t = threadIdx.x; t < by * bz * P; t += w.act) {
      const int f = v.f(w.p, ly, lz), h = f + (2 * lz + v.bym + 3) * P, fy = f + lz * P;
      const int o = (par + ly + lz) & 1;
      const int jl = o ? 0 : dlo, jh = o ? dhi : 0;
      T num = -v.B[C * v.n1 + f];
      if (!zero) {
        num = fma(v.HX[C * v.n1 + f], Xo[h + jl], num);
        num = fma(v.HX[(1 - C) * v.n1 + f + jh], Xo[h + jh], num);
        num = fma(v.HY[C * v.n1y + fy], Xo[h - P], num);
        num = fma(v.HY[(1 - C) * v.n1y + fy + P], Xo[h + P], num);
        num = fma(v.HZ[C * v.n1z + f], Xo[h - sZ], num);
        num = fma(v.HZ[(1 - C) * v.n1z + f + v.bym * P], Xo[h + sZ], num);
      }
      const T x = num * v.ID[C * v.n1 + f];
      Xc[h] = x;
      // boundary rows: to the block beside, or this block's own halo
      if (ly == 0) {
        if (v.py == 1) Xc[h + by * P] = x;
        else if (exchange) ct_send(rem[0] + m + lz * P * W, x, e);
      }
      if (ly == by - 1) {
        if (v.py == 1) Xc[h - by * P] = x;
        else if (exchange) ct_send(rem[1] + m + lz * P * W, x, e);
      }
      if (lz == 0) {
        if (v.pz == 1) Xc[h + bz * sZ] = x;
        else if (exchange) ct_send(rem[2] + m + ly * P * W, x, e);
      }
      if (lz == bz - 1) {
        if (v.pz == 1) Xc[h - bz * sZ] = x;
        else if (exchange) ct_send(rem[3] + m + ly * P * W, x, e);
      }
      ly += w.dly, lz += w.dlz;
      if (ly >= by) ly -= by, ++lz;
    }
  }
  if (exchange) {
    const int ry = v.py > 1 ? 2 * bz : 0, rz = v.pz > 1 ? 2 * by : 0;  // halo rows received
    const int rpt = w.act / P;
    if (w.works)
      for (int row = (threadIdx.x - w.p) / P; row < ry + rz; row += rpt) {
        int slot, dst;
        if (row < ry) {
          const bool hi = row >= bz;
          const int k = hi ? row - bz : row;
          slot = ((hi ? v.bzm : 0) + k) * P + w.p;
          dst = v.h(w.p, hi ? by : -1, k);
        } else {
          const bool hi = row - ry >= by;
          const int j = row - ry - (hi ? by : 0);
          slot = (2 * v.bzm + (hi ? v.bym : 0) + j) * P + w.p;
          dst = v.h(w.p, j, hi ? bz : -1);
        }
        T x = 0;
        bool got = false;
        for (int it = 0; !got && !dead && it < CT_POLL; ++it)
          got = ct_recv(mail + m + slot * W, e, x);
        if (!got) {
          if (!dead) *(volatile double *)err = 1.0;
          dead = true;
        }
        Xc[dst] = x;
      }
  }
  dead = __syncthreads_or(dead) != 0;
}

// residual b - A x at cell (pair p, position o, row ly, plane lz) of the block
// (difference form, op_at's operand order)
template <typename T>
__device__ __forceinline__ T ct_resid(const CtView<T> &v, int p, int o, int ly, int lz) {
  const int c = (v.y0 + v.z0 + ly + lz + o) & 1, P = v.P, sZ = (v.bym + 2) * P;
  const int f = v.f(p, ly, lz), h = v.h(p, ly, lz), fy = f + lz * P;
  const int jl = o ? 0 : (p == 0 ? P - 1 : -1), jh = o ? (p == P - 1 ? 1 - P : 1) : 0;
  const T *Xo = v.X + (1 - c) * v.nh;
  const T xc = v.X[c * v.nh + h];
  T s = v.HX[c * v.n1 + f] * (Xo[h + jl] - xc);
  s = fma(v.HX[(1 - c) * v.n1 + f + jh], Xo[h + jh] - xc, s);
  s = fma(v.HY[c * v.n1y + fy], Xo[h - P] - xc, s);
  s = fma(v.HY[(1 - c) * v.n1y + fy + P], Xo[h + P] - xc, s);
  s = fma(v.HZ[c * v.n1z + f], Xo[h - sZ] - xc, s);
  s = fma(v.HZ[(1 - c) * v.n1z + f + v.bym * P], Xo[h + sZ] - xc, s);
  if (v.DD) s = fma(-v.DD[c * v.n1 + f], xc, s);
  return v.B[c * v.n1 + f] - s;
}

// x ~= At^-1 rhs on the tail's top level (zero initial guess): one symmetric
// V-cycle over every level the cluster holds.  Every CTA takes part in every
// cluster barrier.
template <typename T>
__global__ void __launch_bounds__(CTL_THREADS, 1)
k_ctail(const __grid_constant__ CtArgs<T> a, const T *rhs, T *xout) {
  cgx::cluster_group cl = cgx::this_cluster();
  const int rank = (int)cl.block_rank(), tid = threadIdx.x;
  const int nctas = (int)cl.num_blocks();
  extern __shared__ __align__(16) unsigned char ct_raw[];
  T *base = reinterpret_cast<T *>(ct_raw);
  __shared__ double mean_s;
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(ct_raw);
  const uint32_t mail = sbase + a.mail, flip = a.mail_words * 4;  // half of the words, in bytes
  constexpr int W = sizeof(T) == 8 ? 16 : 8;
  const int last = a.nlev - 1;
  // this CTA's blocks of the level coefficients.  They were formed with the
  // geometry, before the kernel this launch follows: read ahead of the wait
  for (int l = 0; l < last; ++l) {
    const CtLevel<T> &g = a.lv[l];
    const CtView<T> v(base, g, rank);
    if (!v.own) continue;
    const CtWalk w(v.P, v.by + 1);  // rows 0 .. by, planes 0 .. bz: the high faces too
    if (w.works) {
      int ly = w.ly0, lz = w.lz0;
      for (; lz <= v.bz;) {
        const int y = v.y0 + ly == v.ny ? 0 : v.y0 + ly, z = v.z0 + lz == v.nz ? 0 : v.z0 + lz;
        const int q = (v.y0 + ly + v.z0 + lz) & 1;  // colour of the pair's first cell
        const size_t c = at(g.d, 2 * w.p, y, z);
        const bool iny = ly < v.by, inz = lz < v.bz;
        if (inz) {
          const int s = (lz * (v.bym + 1) + ly) * v.P + w.p;
          v.HY[q * v.n1y + s] = g.by[c];
          v.HY[(1 - q) * v.n1y + s] = g.by[c + 1];
        }
        if (iny) {
          const int s = v.f(w.p, ly, lz);
          v.HZ[q * v.n1z + s] = g.bz[c];
          v.HZ[(1 - q) * v.n1z + s] = g.bz[c + 1];
          if (inz) {
            v.HX[q * v.n1 + s] = g.bx[c];
            v.HX[(1 - q) * v.n1 + s] = g.bx[c + 1];
            v.ID[q * v.n1 + s] = g.idiag[c];
            v.ID[(1 - q) * v.n1 + s] = g.idiag[c + 1];
            if (v.DD) {
              v.DD[q * v.n1 + s] = g.dd[c];
              v.DD[(1 - q) * v.n1 + s] = g.dd[c + 1];
            }
          }
        }
        ly += w.dly, lz += w.dlz;
        if (ly >= v.by + 1) ly -= v.by + 1, ++lz;
      }
    }
  }
  for (int e = tid; e < a.mail_words; e += CTL_THREADS)
    reinterpret_cast<unsigned long long *>(ct_raw + a.mail)[e] = 0ull;
  griddep_wait();
  {
    const CtView<T> v(base, a.lv[0], rank);
    if (v.own) {
      const CtWalk w(v.P, v.by);
      if (w.works) {
        int ly = w.ly0, lz = w.lz0;
        for (int t = tid; t < v.by * v.bz * v.P; t += w.act) {
          const int q = (v.y0 + ly + v.z0 + lz) & 1, s = v.f(w.p, ly, lz);
          const size_t c = at(a.lv[0].d, 2 * w.p, v.y0 + ly, v.z0 + lz);
          v.B[q * v.n1 + s] = rhs[c];
          v.B[(1 - q) * v.n1 + s] = rhs[c + 1];
          ly += w.dly, lz += w.dlz;
          if (ly >= v.by) ly -= v.by, ++lz;
        }
      }
    }
  }
  bool dead = *(volatile double *)a.err != 0.0;
  cl.sync();  // every CTA of the cluster has started, loaded its blocks and cleared its slots
  unsigned e = 0;  // epoch of the last exchange, counted alike by every CTA

  // the sweeps of one level: colours c0, 1 - c0; the last exchange of an
  // upward visit is not needed
  auto sweeps = [&](const CtView<T> &v, auto first, int nu, bool zero, bool keep_last) {
    constexpr int C0 = decltype(first)::value;
    if (v.own) {
      const CtWalk w(v.P, v.by);
      uint32_t rem[4];
      const int ym = (v.cy == 0 ? v.py - 1 : v.cy - 1) + v.cz * v.py,
                yp = (v.cy == v.py - 1 ? 0 : v.cy + 1) + v.cz * v.py,
                zm = v.cy + (v.cz == 0 ? v.pz - 1 : v.cz - 1) * v.py,
                zp = v.cy + (v.cz == v.pz - 1 ? 0 : v.cz + 1) * v.py;
      rem[0] = ct_map(mail + (v.bzm * v.P + w.p) * W, ym);
      rem[1] = ct_map(mail + w.p * W, yp);
      rem[2] = ct_map(mail + ((2 * v.bzm + v.bym) * v.P + w.p) * W, zm);
      rem[3] = ct_map(mail + (2 * v.bzm * v.P + w.p) * W, zp);
      for (int s = 0; s < nu; ++s) {
        ct_half<T, C0>(v, w, zero && s == 0, e + 2 * s + 1, mail, rem, flip, dead, a.err);
        const bool x = keep_last || s + 1 < nu;
        ct_half<T, 1 - C0>(v, w, false, x ? e + 2 * s + 2 : 0u, mail, rem, flip, dead, a.err);
      }
    }
    e += 2 * nu;
  };

  for (int l = 0; l < last; ++l) {  // down
    const CtView<T> v(base, a.lv[l], rank);
    sweeps(v, VsColour<0>{}, a.lv[l].nu1, true, true);
    const CtLevel<T> &gc = a.lv[l + 1];
    const bool coarsest = l + 1 == last;
    if (v.own) {  // residual, restricted to the coarser block's owner
      const CtView<T> vc(base, gc, rank);
      const int hy = v.by >> 1;
      const CtWalk w(v.P, hy);
      if (w.works) {
        int J = w.ly0, K = w.lz0;
        for (int t = tid; t < hy * (v.bz >> 1) * v.P; t += w.act) {
          T sum = 0;
#pragma unroll
          for (int q = 0; q < 4; ++q)  // the children of colour 0 (see k_resid_restrict_h)
            sum += ct_resid(v, w.p, (q & 1) ^ (q >> 1), 2 * J + (q & 1), 2 * K + (q >> 1));
          const T r = (T)0.5 * sum;
          const int y = (v.y0 >> 1) + J, z = (v.z0 >> 1) + K;
          if (coarsest) {
            const uint32_t to =
                sbase + (gc.off + gc.n + w.p + gc.d.nx * (y + gc.d.ny * z)) * (int)sizeof(T);
            for (int k = 0; k < nctas; ++k) ct_st(ct_map(to, k), r);
          } else {
            const int oy = ct_part(vc.ny, vc.py, y), oz = ct_part(vc.nz, vc.pz, z);
            const int ly = y - ct_cut(vc.ny, vc.py, oy), lz = z - ct_cut(vc.nz, vc.pz, oz);
            const int c = (w.p + y + z) & 1;
            T *p = vc.B + c * vc.n1 + vc.f(w.p >> 1, ly, lz);
            ct_st(ct_map((uint32_t)__cvta_generic_to_shared(p), oy + oz * vc.py), r);
          }
          J += w.dly, K += w.dlz;
          if (J >= hy) J -= hy, ++K;
        }
      }
    }
    cl.sync();
  }
  {  // coarsest: x = Minv (-(b - mean b)) in FP64, rows spread over the cluster's warps
    const CtLevel<T> &g = a.lv[last];
    const int n = g.n;
    T *X = base + g.off, *B = X + n;
    double acc0 = 0.0;
    for (int q = tid; q < n; q += CTL_THREADS) acc0 += (double)B[q];
    const double sum = block_sum(acc0);
    if (tid == 0) mean_s = a.singular ? sum / n : 0.0;
    __syncthreads();
    const double mean = mean_s;
    const int lane = tid & 31;
    for (int r = rank * (CTL_THREADS / 32) + (tid >> 5); r < n; r += nctas * (CTL_THREADS / 32)) {
      double acc = 0.0;
      for (int c = lane; c < n; c += 32)
        acc = fma(__ldg(a.Minv + (size_t)r * n + c), (double)B[c] - mean, acc);
      const T x = (T)(-warp_sum(acc));
      if (lane < nctas) ct_st(ct_map((uint32_t)__cvta_generic_to_shared(X + r), lane), x);
    }
    cl.sync();
  }
  for (int l = last - 1; l >= 0; --l) {  // up
    const CtView<T> v(base, a.lv[l], rank);
    const CtLevel<T> &gc = a.lv[l + 1];
    if (v.own) {  // the parents' corrections, halo rows included (faces of the block, not corners)
      const CtView<T> vc(base, gc, rank);
      const CtWalk w(v.P, v.by + 2);
      if (w.works) {
        int hy = w.ly0, hz = w.lz0;
        for (; hz < v.bz + 2;) {
          const bool ey = hy == 0 || hy == v.by + 1, ez = hz == 0 || hz == v.bz + 1;
          if (!(ey && ez)) {
            int y = v.y0 + hy - 1, z = v.z0 + hz - 1;
            y = y < 0 ? y + v.ny : (y >= v.ny ? y - v.ny : y);
            z = z < 0 ? z + v.nz : (z >= v.nz ? z - v.nz : z);
            const int J = y >> 1, K = z >> 1;
            T x;
            if (l + 1 == last) {
              x = base[gc.off + w.p + gc.d.nx * (J + gc.d.ny * K)];
            } else {
              const int oy = ct_part(vc.ny, vc.py, J), oz = ct_part(vc.nz, vc.pz, K);
              const int ly = J - ct_cut(vc.ny, vc.py, oy), lz = K - ct_cut(vc.nz, vc.pz, oz);
              const int c = (w.p + J + K) & 1;
              T *p = vc.X + c * vc.nh + vc.h(w.p >> 1, ly, lz);
              x = ct_ld(ct_map((uint32_t)__cvta_generic_to_shared(p), oy + oz * vc.py), T());
            }
            const int s = v.h(w.p, hy - 1, hz - 1);
            v.X[s] += x;
            v.X[v.nh + s] += x;
          }
          hy += w.dly, hz += w.dlz;
          if (hy >= v.by + 2) hy -= v.by + 2, ++hz;
        }
      }
      __syncthreads();
    }
    sweeps(v, VsColour<1>{}, a.lv[l].nu2, false, false);
    if (l > 0) cl.sync();  // the finer level reads this one's x
  }
  const CtView<T> v(base, a.lv[0], rank);
  if (v.own) {
    const CtWalk w(v.P, v.by);
    if (w.works) {
      int ly = w.ly0, lz = w.lz0;
      for (int t = tid; t < v.by * v.bz * v.P; t += w.act) {
        const int q = (v.y0 + ly + v.z0 + lz) & 1, s = v.h(w.p, ly, lz);
        const size_t c = at(a.lv[0].d, 2 * w.p, v.y0 + ly, v.z0 + lz);
        xout[c] = v.X[q * v.nh + s];
        xout[c + 1] = v.X[(1 - q) * v.nh + s];
        ly += w.dly, lz += w.dlz;
        if (ly >= v.by) ly -= v.by, ++lz;
      }
    }
  }
  cl.sync();  // no CTA leaves while another may still write to its shared memory
}

}  // namespace mp
