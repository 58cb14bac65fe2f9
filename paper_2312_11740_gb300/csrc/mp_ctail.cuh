// Coarse tail of the V-cycle on one thread-block cluster (A6-A9).
//
// Below some ten thousand cells every V-cycle kernel is latency-bound: a
// half-sweep of a 16^3 level is a launch of ~2 us whatever its size.  One launch of
// a cluster of up to CT_MAX_CTAS CTAs runs the top level it can take (32^3 at
// 256^3) and every coarser one: sweeps, restrictions, prolongations and the
// coarsest solve.  32^3 to 4^3 under a 256^3 grid: 80 us (108 as z-slabs on 8 CTAs
// with a cluster barrier after every step); a half-sweep of 32^3 takes 0.87 us,
// bound by the warps' issue, of 16^3 and 8^3 0.4.
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
// up sets *err and finishes without waiting (its result is not used).  It still
// sends and is sent to, so the last barrier follows the last exchange of the top
// level in every CTA: none leaves while another may write to its shared memory (about 1 us
// a launch: a 32^3 projection step of 11 iterations takes 1629 us, 1617 with the
// barrier arrived at before the top level's last sweeps, which did not hold this).
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

constexpr int CT_MAX_CTAS = 16, CTL_THREADS = 512, CT_MAX_LEVELS = 10;
constexpr int CT_MAX_TAB = 1024;  // rows and planes of all levels
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
  int polls;       // polls of one wait (CT_POLL)
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

// Quotient t / d from m = ct_magic(d) (round-up reciprocal: exact while t d <
// 2^32).  d = 1 gives m = 0, read as "the quotient is t".
__device__ __forceinline__ unsigned ct_magic(unsigned d) { return 0xFFFFFFFFu / d + 1u; }
__device__ __forceinline__ int ct_div(int t, unsigned m) {
  return m ? (int)__umulhi((unsigned)t, m) : t;
}

// This CTA's part of a level, formed once per launch in shared memory (the
// divisions behind it take about a microsecond and every step of a level
// needs them): block origin and size, neighbours, and the multipliers of the walks.
struct CtBlock {
  int own, cy, cz, y0, by, z0, bz;
  int ym, yp, zm, zp;            // CTAs of the blocks beside
  unsigned mP, mh, m0, m1, m2;   // ct_magic of P, by / 2, by, by + 1, by + 2
};

// One level seen by one CTA.
template <typename T>
struct CtView {
  T *X, *B, *ID, *HX, *HY, *HZ, *DD;
  int nx, ny, nz, P, py, pz, bym, bzm, y0, by, z0, bz;
  int n1, nh, n1y, n1z;
  bool own;  // this CTA holds a block
  __device__ CtView(T *base, const CtLevel<T> &l, const CtBlock &k) {
    nx = l.d.nx, ny = l.d.ny, nz = l.d.nz, P = nx >> 1;
    py = l.py, pz = l.pz, bym = l.bym, bzm = l.bzm;
    own = k.own, y0 = k.y0, by = k.by, z0 = k.z0, bz = k.bz;
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

// The walk of a thread over its cells: one pair p, rows advancing by rpt.  rows:
// rows of a plane of the walk, m its ct_magic.
struct CtWalk {
  int p, act, ly0, lz0, dly, dlz;
  bool works;
  __device__ CtWalk(int P, unsigned mP, int rows, unsigned m) {
    const int tid = threadIdx.x, rpt = ct_div(CTL_THREADS, mP);
    act = rpt * P;
    works = tid < act;
    const int r0 = ct_div(tid, mP);
    p = tid - r0 * P;
    lz0 = ct_div(r0, m), ly0 = r0 - lz0 * rows;
    dlz = ct_div(rpt, m), dly = rpt - dlz * rows;
  }
};

// One colour of one sweep on this CTA's block, and the exchange of its boundary
// rows under epoch e (0: none).  zero: x is taken as zero.  mail: local address of the slots.
template <typename T, int C>
__device__ __forceinline__ void ct_half(const CtView<T> &v, const CtWalk &w, bool zero, unsigned e,
                                        uint32_t mail, const uint32_t rem[4], uint32_t flip,
                                        bool &dead, int polls, double *err) {
  constexpr int W = sizeof(T) == 8 ? 16 : 8;  // bytes of a slot
  const int P = v.P, by = v.by, bz = v.bz, sZ = (v.bym + 2) * P;
  const int dlo = w.p == 0 ? P - 1 : -1, dhi = w.p == P - 1 ? 1 - P : 1;
  const int par = v.y0 + v.z0 + C, ncta = v.py * v.pz;
  const bool exchange = e != 0u && ncta > 1;
  const uint32_t m = (e & 1u) ? flip : 0u;
  T *Xc = v.X + C * v.nh;
  const T *Xo = v.X + (1 - C) * v.nh;
  if (w.works) {
    // two cells at a time: both cells' operands are loaded before either is stored
    // (the compiler cannot move a load past a store to shared memory)
    int ly = w.ly0, lz = w.lz0;
    for (int t = threadIdx.x; t < by * bz * P; t += 2 * w.act) {
      int yy[2], zz[2], hh[2];
      T xx[2];
      const bool two = t + w.act < by * bz * P;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        yy[u] = ly, zz[u] = lz;
        if (u == 0 || two) {
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
          xx[u] = num * v.ID[C * v.n1 + f];
          hh[u] = h;
        }
        ly += w.dly, lz += w.dlz;
        if (ly >= by) ly -= by, ++lz;
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        if (u == 1 && !two) break;
        const T x = xx[u];
        const int h = hh[u], y = yy[u], z = zz[u];
        Xc[h] = x;
        // boundary rows: to the block beside, or this block's own halo
        if (y == 0) {
          if (v.py == 1) Xc[h + by * P] = x;
          else if (exchange) ct_send(rem[0] + m + z * P * W, x, e);
        }
        if (y == by - 1) {
          if (v.py == 1) Xc[h - by * P] = x;
          else if (exchange) ct_send(rem[1] + m + z * P * W, x, e);
        }
        if (z == 0) {
          if (v.pz == 1) Xc[h + bz * sZ] = x;
          else if (exchange) ct_send(rem[2] + m + y * P * W, x, e);
        }
        if (z == bz - 1) {
          if (v.pz == 1) Xc[h - bz * sZ] = x;
          else if (exchange) ct_send(rem[3] + m + y * P * W, x, e);
        }
      }
    }
  }
  if (exchange) {
    const int ry = v.py > 1 ? 2 * bz : 0, rz = v.pz > 1 ? 2 * by : 0;  // halo rows received
    if (w.works)
      for (int row = w.lz0 * by + w.ly0; row < ry + rz; row += w.dlz * by + w.dly) {
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
        for (int it = 0; !got && !dead && it < polls; ++it)
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
  __shared__ CtBlock blk[CT_MAX_LEVELS];
  // owner and local index of every row y and plane z of a level, by level: part << 16 | local
  __shared__ int tab[CT_MAX_TAB], tab0[CT_MAX_LEVELS];
  const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(ct_raw);
  const uint32_t mail = sbase + a.mail, flip = a.mail_words * 4;  // half of the words, in bytes
  constexpr int W = sizeof(T) == 8 ? 16 : 8;
  const int last = a.nlev - 1;
  // Nothing up to the wait depends on the kernel this launch follows (the level
  // coefficients were formed with the geometry), so it overlaps that kernel's end.
  if (tid < last) {
    const CtLevel<T> &g = a.lv[tid];
    CtBlock k;
    k.own = rank < g.py * g.pz;
    k.cy = k.own ? rank % g.py : 0, k.cz = k.own ? rank / g.py : 0;
    k.y0 = ct_cut(g.d.ny, g.py, k.cy), k.by = ct_cut(g.d.ny, g.py, k.cy + 1) - k.y0;
    k.z0 = ct_cut(g.d.nz, g.pz, k.cz), k.bz = ct_cut(g.d.nz, g.pz, k.cz + 1) - k.z0;
    k.ym = (k.cy == 0 ? g.py - 1 : k.cy - 1) + k.cz * g.py;
    k.yp = (k.cy == g.py - 1 ? 0 : k.cy + 1) + k.cz * g.py;
    k.zm = k.cy + (k.cz == 0 ? g.pz - 1 : k.cz - 1) * g.py;
    k.zp = k.cy + (k.cz == g.pz - 1 ? 0 : k.cz + 1) * g.py;
    k.mP = ct_magic(g.d.nx >> 1), k.mh = ct_magic(k.by >> 1), k.m0 = ct_magic(k.by);
    k.m1 = ct_magic(k.by + 1), k.m2 = ct_magic(k.by + 2);
    blk[tid] = k;
    int t0 = 0;
    for (int l = 0; l < tid; ++l) t0 += a.lv[l].d.ny + a.lv[l].d.nz;
    tab0[tid] = t0;
  }
  for (int e = tid; e < a.mail_words; e += CTL_THREADS)
    reinterpret_cast<unsigned long long *>(ct_raw + a.mail)[e] = 0ull;
  __syncthreads();
  for (int l = 1; l < last; ++l) {
    const CtLevel<T> &g = a.lv[l];
    for (int q = tid; q < g.d.ny + g.d.nz; q += CTL_THREADS) {
      const bool y = q < g.d.ny;
      const int n = y ? g.d.ny : g.d.nz, p = y ? g.py : g.pz, row = y ? q : q - g.d.ny;
      const int c = ct_part(n, p, row);
      tab[tab0[l] + q] = c << 16 | (row - ct_cut(n, p, c));
    }
  }
  for (int l = 0; l < last; ++l) {  // this CTA's blocks of the level coefficients
    const CtLevel<T> &g = a.lv[l];
    const CtView<T> v(base, g, blk[l]);
    if (!v.own) continue;
    const CtWalk w(v.P, blk[l].mP, v.by + 1, blk[l].m1);  // rows 0 .. by, planes 0 .. bz
    if (w.works) {
      int ly = w.ly0, lz = w.lz0;
      for (; lz <= v.bz;) {
        const int y = v.y0 + ly == v.ny ? 0 : v.y0 + ly, z = v.z0 + lz == v.nz ? 0 : v.z0 + lz;
        const int q = (v.y0 + ly + v.z0 + lz) & 1;  // colour of the pair's first cell
        const size_t c = at(g.d, 2 * w.p, y, z);
        const bool iny = ly < v.by, inz = lz < v.bz;
        if (inz) {
          const int s = (lz * (v.bym + 1) + ly) * v.P + w.p;
          const auto fy = vs_pair(g.by + c);
          v.HY[q * v.n1y + s] = fy.x;
          v.HY[(1 - q) * v.n1y + s] = fy.y;
        }
        if (iny) {
          const int s = v.f(w.p, ly, lz);
          const auto fz = vs_pair(g.bz + c);
          if (inz) {
            const auto fx = vs_pair(g.bx + c), id = vs_pair(g.idiag + c);
            v.HX[q * v.n1 + s] = fx.x;
            v.HX[(1 - q) * v.n1 + s] = fx.y;
            v.ID[q * v.n1 + s] = id.x;
            v.ID[(1 - q) * v.n1 + s] = id.y;
            if (v.DD) {
              const auto dd = vs_pair(g.dd + c);
              v.DD[q * v.n1 + s] = dd.x;
              v.DD[(1 - q) * v.n1 + s] = dd.y;
            }
          }
          v.HZ[q * v.n1z + s] = fz.x;
          v.HZ[(1 - q) * v.n1z + s] = fz.y;
        }
        ly += w.dly, lz += w.dlz;
        if (ly >= v.by + 1) ly -= v.by + 1, ++lz;
      }
    }
  }
  cl.sync();  // every CTA of the cluster has started and cleared its slots
  griddep_wait();
  {
    const CtView<T> v(base, a.lv[0], blk[0]);
    if (v.own) {
      const CtWalk w(v.P, blk[0].mP, v.by, blk[0].m0);
      if (w.works) {
        int ly = w.ly0, lz = w.lz0;
        for (int t = tid; t < v.by * v.bz * v.P; t += w.act) {
          const int q = (v.y0 + ly + v.z0 + lz) & 1, s = v.f(w.p, ly, lz);
          const auto r = vs_pair(rhs + at(a.lv[0].d, 2 * w.p, v.y0 + ly, v.z0 + lz));
          v.B[q * v.n1 + s] = r.x;
          v.B[(1 - q) * v.n1 + s] = r.y;
          ly += w.dly, lz += w.dlz;
          if (ly >= v.by) ly -= v.by, ++lz;
        }
      }
    }
  }
  bool dead = *(volatile double *)a.err != 0.0;
  __syncthreads();
  unsigned e = 0;  // epoch of the last exchange, counted alike by every CTA

  // the sweeps of one level: colours c0, 1 - c0; the last exchange of an
  // upward visit is not needed.  leave (the kernel's last sweeps): arrive at the
  // last cluster barrier once this CTA has sent and received everything, which
  // leaves the last half-sweep to cover the other CTAs' arrival
  auto sweeps = [&](const CtView<T> &v, const CtBlock &k, auto first, int nu, bool zero,
                    bool keep_last, bool leave) {
    constexpr int C0 = decltype(first)::value;
    if (v.own) {
      const CtWalk w(v.P, k.mP, v.by, k.m0);
      uint32_t rem[4];
      rem[0] = ct_map(mail + (v.bzm * v.P + w.p) * W, k.ym);
      rem[1] = ct_map(mail + w.p * W, k.yp);
      rem[2] = ct_map(mail + ((2 * v.bzm + v.bym) * v.P + w.p) * W, k.zm);
      rem[3] = ct_map(mail + (2 * v.bzm * v.P + w.p) * W, k.zp);
      for (int s = 0; s < nu; ++s) {
        ct_half<T, C0>(v, w, zero && s == 0, e + 2 * s + 1, mail, rem, flip, dead, a.polls, a.err);
        const bool x = keep_last || s + 1 < nu;
        if (leave && s + 1 == nu) cl.barrier_arrive();
        ct_half<T, 1 - C0>(v, w, false, x ? e + 2 * s + 2 : 0u, mail, rem, flip, dead, a.polls,
                           a.err);
      }
    } else if (leave) {
      cl.barrier_arrive();
    }
    e += 2 * nu;
  };

  for (int l = 0; l < last; ++l) {  // down
    const CtView<T> v(base, a.lv[l], blk[l]);
    sweeps(v, blk[l], VsColour<0>{}, a.lv[l].nu1, true, true, false);
    const CtLevel<T> &gc = a.lv[l + 1];
    const bool coarsest = l + 1 == last;
    if (v.own) {  // residual, restricted to the coarser block's owner
      const CtView<T> vc(base, gc, blk[coarsest ? l : l + 1]);
      const int *ty = tab + tab0[coarsest ? l : l + 1], *tz = ty + vc.ny;
      const int hy = v.by >> 1;
      const CtWalk w(v.P, blk[l].mP, hy, blk[l].mh);
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
            const int ey = ty[y], ez = tz[z], c = (w.p + y + z) & 1;
            T *p = vc.B + c * vc.n1 + vc.f(w.p >> 1, ey & 0xffff, ez & 0xffff);
            ct_st(ct_map((uint32_t)__cvta_generic_to_shared(p), (ey >> 16) + (ez >> 16) * vc.py), r);
          }
          J += w.dly, K += w.dlz;
          if (J >= hy) J -= hy, ++K;
        }
      }
    }
    cl.sync();
  }
  {  // coarsest: x = -Minv (b - mean b) in FP64, rows spread over the cluster's warps.
    // Minv 1 = 1 for a singular operator (M 1 = 1), so the mean is added to the
    // product instead of removed from b, and every warp forms it along the way
    const CtLevel<T> &g = a.lv[last];
    const int n = g.n;
    T *X = base + g.off, *B = X + n;
    const int lane = tid & 31;
    for (int r = rank * (CTL_THREADS / 32) + (tid >> 5); r < n; r += nctas * (CTL_THREADS / 32)) {
      double acc = 0.0, sum = 0.0;
#pragma unroll 4
      for (int c = lane; c < n; c += 32) {
        const double bc = (double)B[c];
        acc = fma(__ldg(a.Minv + (size_t)r * n + c), bc, acc);
        sum += bc;
      }
      acc = warp_sum(acc);
      sum = a.singular ? warp_sum(sum) / n : 0.0;
      if (lane < nctas) ct_st(ct_map((uint32_t)__cvta_generic_to_shared(X + r), lane), (T)(sum - acc));
    }
    cl.sync();
  }
  for (int l = last - 1; l >= 0; --l) {  // up
    const CtView<T> v(base, a.lv[l], blk[l]);
    const CtLevel<T> &gc = a.lv[l + 1];
    if (v.own) {  // the parents' corrections, halo rows included (faces of the block, not corners)
      const int lc = l + 1 == last ? l : l + 1;
      const CtView<T> vc(base, gc, blk[lc]);
      const int *ty = tab + tab0[lc], *tz = ty + vc.ny;
      const CtWalk w(v.P, blk[l].mP, v.by + 2, blk[l].m2);
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
              const int ey2 = ty[J], ez2 = tz[K], c = (w.p + J + K) & 1;
              T *p = vc.X + c * vc.nh + vc.h(w.p >> 1, ey2 & 0xffff, ez2 & 0xffff);
              x = ct_ld(ct_map((uint32_t)__cvta_generic_to_shared(p),
                               (ey2 >> 16) + (ez2 >> 16) * vc.py), T());
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
    sweeps(v, blk[l], VsColour<1>{}, a.lv[l].nu2, false, false, l == 0);
    if (l > 0) cl.sync();  // the finer level reads this one's x
  }
  const CtView<T> v(base, a.lv[0], blk[0]);
  if (v.own) {
    const CtWalk w(v.P, blk[0].mP, v.by, blk[0].m0);
    if (w.works) {
      int ly = w.ly0, lz = w.lz0;
      for (int t = tid; t < v.by * v.bz * v.P; t += w.act) {
        const int q = (v.y0 + ly + v.z0 + lz) & 1, s = v.h(w.p, ly, lz);
        const size_t c = at(a.lv[0].d, 2 * w.p, v.y0 + ly, v.z0 + lz);
        vs_put(xout + c, v.X[q * v.nh + s], v.X[(1 - q) * v.nh + s]);
        ly += w.dly, lz += w.dlz;
        if (ly >= v.by) ly -= v.by, ++lz;
      }
    }
  }
  cl.barrier_wait();  // every CTA is past its last access to another's shared memory
}

}  // namespace mp
