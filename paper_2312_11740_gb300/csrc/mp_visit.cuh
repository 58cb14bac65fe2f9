// One visit of a V-cycle level in one launch: every red-black sweep of the
// visit, with the residual + restriction behind a downward visit and the
// prolongation in front of an upward one (A6-A8).
//
// What bounds the levels between the finest and the coarse tail is latency: as
// one launch per sweep a 64^3 level took ~8 us a sweep and a 128^3 one ~19,
// whatever they moved.  A level whose iterate, right-hand side and face
// coefficients fit the chip's shared memory (FP32 to about 2.1 M cells, of which the
// dispatch takes those up to VISIT_TOP32; FP64 to about 0.6 M, all taken) is
// read once, swept in shared memory and written once.  64^3 FP32:
// 1.37 us a half-sweep and ~5 us a launch; under 256^3 64 us per V-cycle for
// the level's two visits, transfers included (167 for its sweeps alone before).
//
// Blocks: the level is cut in y and z (whole x rows) into py x pz blocks, one
// CTA each, at most one CTA per SM, launched cooperatively: the CTAs wait on
// one another.  A cut lies at even y and z, so the eight children of a coarse
// cell share a block.  After each half-sweep a CTA sends the new values of its
// boundary rows to the up to four blocks beside it and waits for theirs.
//
// The exchange carries no separate flag: a value travels as one 8-byte word
// with the epoch of its half-sweep (FP64: two such words), written and polled
// with relaxed 8-byte accesses, so a round trip through L2 is its whole
// latency.  A slot is reused after two half-sweeps; by then its reader has sent
// its own next message, hence consumed it.  Epochs count on from launch to
// launch (the last CTA to finish stores the next base), so a word of an earlier
// launch never matches.  Every wait is bounded: a CTA that gives up sets *err and
// returns, and later visits return at once.
//
// Shared-memory arrays are split by colour: [colour][row][pair], pair p of a
// row holding cells 2p and 2p + 1, one of each colour.  All six neighbours of
// a cell are of the other colour, at the same pair (y, z) or at the same and
// one next pair (x): every access of a half-sweep has unit stride.
//
// Same arithmetic as the per-level launches, operation for operation
// (rbgs_h_val / rbgs_cell, resid_h / resid_at, k_prolong): bitwise their
// result.
#pragma once

namespace mp {

constexpr int VS_THREADS = 512;
constexpr int VS_POLL = 1 << 20;  // polls of one wait (about a second)
constexpr int VS_BATCH = 4;       // halo words of a thread in flight at once

template <typename T> struct VsFace { using F = double; };
template <> struct VsFace<float> { using F = __half; };

template <typename T>
struct VisitArgs {
  using F = typename VsFace<T>::F;
  T *x;          // iterate (up: corrected by ec first; down: zero before)
  const T *rhs;  // right-hand side of the level
  const F *hx, *hy, *hz;  // faces (FP32: FP16, scaled by fs)
  const F *dd;            // FP32: outflow diagonal (see dd_h) or null
  const T *idiag, *diag;  // FP64: 1/diag and diag (diag holds the outflow part)
  const T *ec;            // up: the coarser level's iterate
  T *bc;                  // down: the coarser level's right-hand side
  Dims d, dc;
  int nu;                 // sweeps
  int py, pz, bym, bzm;   // blocks, and the largest block's rows and planes
  float fs, inv_fs;
  unsigned long long *mail;  // exchange slots
  unsigned *epoch;           // [0] base of this launch, [1] CTAs done
  int polls;                 // polls of one wait (VS_POLL)
  double *err;               // set when a wait gave up
};

// exchange slots of one CTA and parity: y-low, y-high (planes x pairs),
// z-low, z-high (rows x pairs)
__host__ __device__ inline size_t vs_slots(int nx, int bym, int bzm) {
  return (size_t)(bym + bzm) * nx;  // 2 (bym + bzm) (nx / 2)
}
template <typename T>
__host__ __device__ constexpr int vs_words() { return sizeof(T) == 8 ? 2 : 1; }

// shared memory of a block of by x bz rows: x with its halo, faces, 1/diag
// and b (FP64), outflow diagonal
template <typename T>
inline size_t vs_smem(int nx, int by, int bz, bool dd) {
  using F = typename VsFace<T>::F;
  const size_t own = (size_t)by * bz * nx;
  size_t s = sizeof(T) * (size_t)(by + 2) * (bz + 2) * nx;
  s += sizeof(T) * own * (sizeof(T) == 8 ? 2 : 1);
  s += sizeof(F) * (own + (size_t)(by + 1) * bz * nx + (size_t)by * (bz + 1) * nx);
  if (dd) s += sizeof(F) * own;
  return s + 16;
}

__device__ __forceinline__ void vs_st(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long vs_ld(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void vs_send(unsigned long long *slot, float v, unsigned epoch) {
  vs_st(slot, ((unsigned long long)epoch << 32) | __float_as_uint(v));
}
__device__ __forceinline__ void vs_send(unsigned long long *slot, double v, unsigned epoch) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(v);
  vs_st(slot, ((unsigned long long)epoch << 32) | (u & 0xffffffffull));
  vs_st(slot + 1, ((unsigned long long)epoch << 32) | (u >> 32));
}
// the words of one slot, and the value in them once they carry this epoch
struct VsWord1 {
  unsigned long long a;
  __device__ void load(const unsigned long long *slot) { a = vs_ld(slot); }
  __device__ bool holds(unsigned epoch) const { return (unsigned)(a >> 32) == epoch; }
  __device__ float value() const { return __uint_as_float((unsigned)a); }
};
struct VsWord2 {
  unsigned long long a, b;
  __device__ void load(const unsigned long long *slot) { a = vs_ld(slot), b = vs_ld(slot + 1); }
  __device__ bool holds(unsigned epoch) const {
    return (unsigned)(a >> 32) == epoch && (unsigned)(b >> 32) == epoch;
  }
  __device__ double value() const {
    return __longlong_as_double((long long)((a & 0xffffffffull) | (b << 32)));
  }
};
template <typename T> struct VsWord { using W = VsWord2; };
template <> struct VsWord<float> { using W = VsWord1; };

__device__ __forceinline__ float vs_f(__half v) { return __half2float(v); }
__device__ __forceinline__ double vs_f(double v) { return v; }

// two consecutive elements of a row (even index: aligned to the pair)
struct VsH2 { __half x, y; };
__device__ __forceinline__ float2 vs_pair(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ double2 vs_pair(const double *p) { return *reinterpret_cast<const double2 *>(p); }
__device__ __forceinline__ VsH2 vs_pair(const __half *p) {
  const __half2 h = *reinterpret_cast<const __half2 *>(p);
  return VsH2{__low2half(h), __high2half(h)};
}
__device__ __forceinline__ void vs_put(float *p, float a, float b) {
  *reinterpret_cast<float2 *>(p) = make_float2(a, b);
}
__device__ __forceinline__ void vs_put(double *p, double a, double b) {
  *reinterpret_cast<double2 *>(p) = make_double2(a, b);
}

template <int C> struct VsColour { static constexpr int value = C; };

// round-up reciprocal division (t d < 2^32; see ct_div)
struct VsDiv {
  unsigned m, d;
  __device__ explicit VsDiv(int dd) : m(dd > 1 ? 0xFFFFFFFFu / (unsigned)dd + 1u : 0u), d(dd) {}
  __device__ int q(int t) const { return m ? (int)__umulhi((unsigned)t, m) : t; }
};

// the operands around cell (row r of the block, pair p, colour c, position o
// in the pair): indices into the colour-split arrays
struct VsAt {
  int f, fxh, fy, fyh, fz, fzh;   // own faces and the high ones
  int xc, xl, xh, yl, yh, zl, zh;  // x of the cell and its neighbours
};
__device__ __forceinline__ VsAt vs_at(int r, int ly, int lz, int p, int o, int P, int by) {
  VsAt a;
  const int pn = o ? (p + 1 == P ? 0 : p + 1) : p;   // pair of the x-high neighbour
  const int pv = o ? p : (p == 0 ? P - 1 : p - 1);   // pair of the x-low neighbour
  const int hr = ((lz + 1) * (by + 2) + ly + 1) * P;
  a.f = r * P + p;
  a.fxh = r * P + pn;
  a.fy = (lz * (by + 1) + ly) * P + p;
  a.fyh = a.fy + P;
  a.fz = a.f;
  a.fzh = a.f + by * P;
  a.xc = hr + p;
  a.xl = hr + pv;
  a.xh = hr + pn;
  a.yl = a.xc - P;
  a.yh = a.xc + P;
  a.zl = a.xc - (by + 2) * P;
  a.zh = a.xc + (by + 2) * P;
  return a;
}

template <typename T, bool UP>
__global__ void __launch_bounds__(VS_THREADS, 1) k_visit(const VisitArgs<T> a) {
  using F = typename VsFace<T>::F;
  griddep_wait();
  extern __shared__ __align__(16) unsigned char vs_raw[];
  if (*(volatile double *)a.err != 0.0) return;
  const unsigned base = *(volatile unsigned *)a.epoch;
  const int tid = threadIdx.x, nx = a.d.nx, ny = a.d.ny, nz = a.d.nz, P = nx >> 1;
  const int py = a.py, pz = a.pz, cy = blockIdx.x % py, cz = blockIdx.x / py;
  const int y0 = 2 * (cy * (ny >> 1) / py), by = 2 * ((cy + 1) * (ny >> 1) / py) - y0;
  const int z0 = 2 * (cz * (nz >> 1) / pz), bz = 2 * ((cz + 1) * (nz >> 1) / pz) - z0;
  const int n1 = by * bz * P;                    // cells of one colour
  const int nh = (by + 2) * (bz + 2) * P;        // with the halo
  const int n1y = (by + 1) * bz * P, n1z = by * (bz + 1) * P;
  T *X = reinterpret_cast<T *>(vs_raw);
  T *B = X + 2 * nh;
  T *ID = B + 2 * n1;
  F *HX = reinterpret_cast<F *>(sizeof(T) == 8 ? ID + 2 * n1 : ID);
  F *HY = HX + 2 * n1, *HZ = HY + 2 * n1y, *DD = HZ + 2 * n1z;
  const VsDiv dP(P), dby(by);

  // ---- the block's arrays
#pragma unroll 2
  for (int t = tid; t < n1; t += VS_THREADS) {
    const int r = dP.q(t), p = t - r * P, lz = dby.q(r), ly = r - lz * by;
    const int q = (y0 + ly + z0 + lz) & 1;  // colour of the pair's first cell
    const size_t g = at(a.d, 2 * p, y0 + ly, z0 + lz);
    const int s0 = q * n1 + t, s1 = (1 - q) * n1 + t;
    const auto fx = vs_pair(a.hx + g), fy = vs_pair(a.hy + g), fz = vs_pair(a.hz + g);
    const auto b = vs_pair(a.rhs + g);
    B[s0] = b.x;
    B[s1] = b.y;
    if constexpr (sizeof(T) == 8) {
      const auto v = vs_pair(a.idiag + g);
      ID[s0] = v.x;
      ID[s1] = v.y;
    }
    if (UP) {
      const auto v = vs_pair(a.x + g);
      const T e = a.ec[at(a.dc, p, (y0 + ly) >> 1, (z0 + lz) >> 1)];
      const int h = ((lz + 1) * (by + 2) + ly + 1) * P + p;
      X[q * nh + h] = v.x + e;
      X[(1 - q) * nh + h] = v.y + e;
    }
    if (sizeof(T) == 4 && a.dd) {
      const auto v = vs_pair(a.dd + g);
      DD[s0] = v.x;
      DD[s1] = v.y;
    }
    HX[s0] = fx.x;
    HX[s1] = fx.y;
    const int ty = (lz * (by + 1) + ly) * P + p;
    HY[q * n1y + ty] = fy.x;
    HY[(1 - q) * n1y + ty] = fy.y;
    HZ[q * n1z + t] = fz.x;
    HZ[(1 - q) * n1z + t] = fz.y;
  }
  const int yw = y0 + by == ny ? 0 : y0 + by, zw = z0 + bz == nz ? 0 : z0 + bz;
  for (int t = tid; t < bz * P; t += VS_THREADS) {  // the y faces above the block
    const int lz = dP.q(t), p = t - lz * P, q = (y0 + by + z0 + lz) & 1;
    const auto v = vs_pair(a.hy + at(a.d, 2 * p, yw, z0 + lz));
    const int s = (lz * (by + 1) + by) * P + p;
    HY[q * n1y + s] = v.x;
    HY[(1 - q) * n1y + s] = v.y;
  }
  for (int t = tid; t < by * P; t += VS_THREADS) {  // the z faces above it
    const int ly = dP.q(t), p = t - ly * P, q = (y0 + ly + z0 + bz) & 1;
    const auto v = vs_pair(a.hz + at(a.d, 2 * p, y0 + ly, zw));
    const int s = bz * by * P + t;
    HZ[q * n1z + s] = v.x;
    HZ[(1 - q) * n1z + s] = v.y;
  }
  if (UP) {  // x of the rows around the block
    for (int t = tid; t < 2 * (by + bz) * P; t += VS_THREADS) {
      const int row = dP.q(t), p = t - row * P;
      int hy, hz;  // halo row: block row + 1
      if (row < 2 * bz) {
        hy = row < bz ? 0 : by + 1;
        hz = (row < bz ? row : row - bz) + 1;
      } else {
        const int w = row - 2 * bz;
        hz = w < by ? 0 : bz + 1;
        hy = (w < by ? w : w - by) + 1;
      }
      int y = y0 + hy - 1, z = z0 + hz - 1;
      const int q = (y + z) & 1;
      y = y < 0 ? y + ny : (y >= ny ? y - ny : y);
      z = z < 0 ? z + nz : (z >= nz ? z - nz : z);
      const auto v = vs_pair(a.x + at(a.d, 2 * p, y, z));
      const T e = a.ec[at(a.dc, p, y >> 1, z >> 1)];
      const int h = (hz * (by + 2) + hy) * P + p;
      X[q * nh + h] = v.x + e;
      X[(1 - q) * nh + h] = v.y + e;
    }
  }
  __syncthreads();

  // ---- half-sweeps.  A thread keeps one pair index p and walks rows: its cell
  // t (+ act per step) of each colour, so indices advance by additions.
  const int rpt = VS_THREADS / P, act = rpt * P;  // rows per step; threads at work
  const bool works = tid < act;
  const int r0 = dP.q(tid), p = tid - r0 * P;
  const int lz0 = dby.q(r0), ly0 = r0 - lz0 * by, dlz = dby.q(rpt), dly = rpt - dlz * by;
  const int sP = P, sZ = (by + 2) * P, sFz = by * P, sY = by * P, sZZ = bz * (by + 2) * P;
  const int dlo = p == 0 ? P - 1 : -1, dhi = p == P - 1 ? 1 - P : 1;  // next pairs in the row
  const int par0 = y0 + z0;
  const size_t slots = vs_slots(nx, a.bym, a.bzm);
  const int ncta = py * pz;
  constexpr int W = vs_words<T>();
  const int fy1 = a.bzm * P, fz0 = 2 * fy1, fz1 = fz0 + a.bym * P;
  const int c_ym = (cy == 0 ? py - 1 : cy - 1) + cz * py, c_yp = (cy == py - 1 ? 0 : cy + 1) + cz * py;
  const int c_zm = cy + (cz == 0 ? pz - 1 : cz - 1) * py, c_zp = cy + (cz == pz - 1 ? 0 : cz + 1) * py;
  const size_t flip = ncta * slots * W;  // from the even epochs' slots to the odd ones'
  unsigned long long *const s_ym = a.mail + (c_ym * slots + fy1 + p) * W;
  unsigned long long *const s_yp = a.mail + (c_yp * slots + p) * W;
  unsigned long long *const s_zm = a.mail + (c_zm * slots + fz1 + p) * W;
  unsigned long long *const s_zp = a.mail + (c_zp * slots + fz0 + p) * W;
  const int rx_y = py > 1 ? 2 * bz : 0, rx_z = pz > 1 ? 2 * by : 0;  // halo rows received
  const int nhalf = 2 * a.nu;
  // one cell: its new value, stored here, in this block's own halo where the block
  // spans the axis, and sent to the block beside where it lies on a boundary row
  auto cell = [&](int c, int t, int ly, int lz, T bv, bool zero, bool exchange, unsigned e,
                  size_t m) {
    const int o = (par0 + ly + lz + c) & 1;
    T *xc = X + c * nh + (t + (2 * lz + by + 3) * sP);
    const T *xo = X + (1 - c) * nh + (t + (2 * lz + by + 3) * sP);
    const F *hxc = HX + c * n1 + t, *hxo = HX + (1 - c) * n1 + t;
    const F *hyc = HY + c * n1y + (t + lz * sP), *hyo = HY + (1 - c) * n1y + (t + lz * sP + sP);
    const F *hzc = HZ + c * n1z + t, *hzo = HZ + (1 - c) * n1z + t + sFz;
    const int jl = o ? 0 : dlo, jh = o ? dhi : 0;
    T v;
    if constexpr (sizeof(T) == 4) {
      const float wxl = vs_f(*hxc), wxh = vs_f(hxo[jh]), wyl = vs_f(*hyc), wyh = vs_f(*hyo),
                  wzl = vs_f(*hzc), wzh = vs_f(*hzo);
      float s = -bv * a.fs;
      if (!zero) {
        s = fmaf(wxl, xo[jl], s);
        s = fmaf(wxh, xo[jh], s);
        s = fmaf(wyl, xo[-sP], s);
        s = fmaf(wyh, xo[sP], s);
        s = fmaf(wzl, xo[-sZ], s);
        s = fmaf(wzh, xo[sZ], s);
      }
      float den = ((wxl + wxh) + (wyl + wyh)) + (wzl + wzh);
      if (a.dd) den += 4.f * vs_f(DD[c * n1 + t]);
      v = __fdividef(s, den);
    } else {
      double s = -bv;
      if (!zero) {
        s = fma(*hxc, xo[jl], s);
        s = fma(hxo[jh], xo[jh], s);
        s = fma(*hyc, xo[-sP], s);
        s = fma(*hyo, xo[sP], s);
        s = fma(*hzc, xo[-sZ], s);
        s = fma(*hzo, xo[sZ], s);
      }
      v = s * ID[c * n1 + t];
    }
    *xc = v;
    if (ly == 0) {
      if (py == 1) xc[sY] = v;
      else if (exchange) vs_send(s_ym + (m + lz * sP * W), v, e);
    }
    if (ly == by - 1) {
      if (py == 1) xc[-sY] = v;
      else if (exchange) vs_send(s_yp + (m + lz * sP * W), v, e);
    }
    if (lz == 0) {
      if (pz == 1) xc[sZZ] = v;
      else if (exchange) vs_send(s_zm + (m + ly * sP * W), v, e);
    }
    if (lz == bz - 1) {
      if (pz == 1) xc[-sZZ] = v;
      else if (exchange) vs_send(s_zp + (m + ly * sP * W), v, e);
    }
  };
  auto half = [&](auto colour, int hs) -> bool {
    constexpr int c = decltype(colour)::value;
    const bool zero = !UP && hs == 0, exchange = ncta > 1 && !(UP && hs == nhalf - 1);
    const unsigned e = base + 1u + (unsigned)hs;
    const size_t m = (e & 1u) ? flip : 0;
    T *xc = X + c * nh;
    int ly = ly0, lz = lz0;
    if (works) {
#pragma unroll 2
      for (int t = tid; t < n1; t += act) {
        cell(c, t, ly, lz, B[c * n1 + t], zero, exchange, e, m);
        ly += dly, lz += dlz;
        if (ly >= by) ly -= by, ++lz;
      }
    }
    bool fail = false;
    if (exchange) {
      const unsigned long long *mine = a.mail + m + blockIdx.x * slots * W;
      const int total = (rx_y + rx_z) * P;
      for (int t0 = tid; t0 < total; t0 += VS_THREADS * VS_BATCH) {
        const unsigned long long *src[VS_BATCH];
        int dst[VS_BATCH];
        typename VsWord<T>::W w[VS_BATCH];
        unsigned wait = 0;
#pragma unroll
        for (int u = 0; u < VS_BATCH; ++u) {
          const int t = t0 + u * VS_THREADS;
          src[u] = mine;
          dst[u] = 0;
          if (t >= total) continue;
          wait |= 1u << u;
          const int row = dP.q(t), q = t - row * P;
          if (row < rx_y) {
            const bool hi = row >= bz;
            const int k = hi ? row - bz : row;
            src[u] = mine + ((hi ? fy1 : 0) + k * P + q) * W;
            dst[u] = ((k + 1) * (by + 2) + (hi ? by + 1 : 0)) * P + q;
          } else {
            const bool hi = row - rx_y >= by;
            const int j = row - rx_y - (hi ? by : 0);
            src[u] = mine + ((hi ? fz1 : fz0) + j * P + q) * W;
            dst[u] = ((hi ? bz + 1 : 0) * (by + 2) + j + 1) * P + q;
          }
        }
        for (int it = 0; wait && it < a.polls; ++it) {
#pragma unroll
          for (int u = 0; u < VS_BATCH; ++u) w[u].load(src[u]);
#pragma unroll
          for (int u = 0; u < VS_BATCH; ++u)
            if (((wait >> u) & 1u) && w[u].holds(e)) {
              xc[dst[u]] = w[u].value();
              wait &= ~(1u << u);
            }
        }
        fail = fail || wait != 0;
      }
    }
    return __syncthreads_or(fail) != 0;
  };
  for (int hs = 0; hs < nhalf; hs += 2)
    if (half(VsColour<UP ? 1 : 0>{}, hs) || half(VsColour<UP ? 0 : 1>{}, hs + 1)) {
      if (tid == 0) *(volatile double *)a.err = 1.0;
      return;
    }

  // ---- the iterate, and behind a downward visit the coarser right-hand side
  for (int t = tid; t < n1; t += VS_THREADS) {
    const int r = dP.q(t), p = t - r * P, lz = dby.q(r), ly = r - lz * by;
    const int q = (y0 + ly + z0 + lz) & 1;
    const int h = ((lz + 1) * (by + 2) + ly + 1) * P + p;
    vs_put(a.x + at(a.d, 2 * p, y0 + ly, z0 + lz), X[q * nh + h], X[(1 - q) * nh + h]);
  }
  if (!UP) {
    const int hy = by >> 1, nc = hy * (bz >> 1) * P;
    const VsDiv dhy(hy);
    for (int t = tid; t < nc; t += VS_THREADS) {
      const int rc = dP.q(t), p = t - rc * P, K = dhy.q(rc), J = rc - K * hy;
      T sum = 0;
#pragma unroll
      for (int w = 0; w < 4; ++w) {  // the children of colour 0
        constexpr int k = 0;
        const int o = (w & 1) ^ (w >> 1), ly = 2 * J + (w & 1), lz = 2 * K + (w >> 1);
        const int r = lz * by + ly;
        const VsAt i = vs_at(r, ly, lz, p, o, P, by);
        const T *xo = X + (1 - k) * nh;
        const F *hxc = HX + k * n1, *hxo = HX + (1 - k) * n1, *hyc = HY + k * n1y,
                *hyo = HY + (1 - k) * n1y, *hzc = HZ + k * n1z, *hzo = HZ + (1 - k) * n1z;
        const T xv = X[k * nh + i.xc];
        const T bv = B[k * n1 + i.f];
        if constexpr (sizeof(T) == 4) {
          float s = vs_f(hxc[i.f]) * (xo[i.xl] - xv);
          s = fmaf(vs_f(hxo[i.fxh]), xo[i.xh] - xv, s);
          s = fmaf(vs_f(hyc[i.fy]), xo[i.yl] - xv, s);
          s = fmaf(vs_f(hyo[i.fyh]), xo[i.yh] - xv, s);
          s = fmaf(vs_f(hzc[i.fz]), xo[i.zl] - xv, s);
          s = fmaf(vs_f(hzo[i.fzh]), xo[i.zh] - xv, s);
          if (a.dd) s = fmaf(-(4.f * vs_f(DD[k * n1 + i.f])), xv, s);
          sum += bv - s * a.inv_fs;
        } else {
          double s = -a.diag[at(a.d, 2 * p + o, y0 + ly, z0 + lz)] * xv;
          s = fma(hxc[i.f], xo[i.xl], s);
          s = fma(hxo[i.fxh], xo[i.xh], s);
          s = fma(hyc[i.fy], xo[i.yl], s);
          s = fma(hyo[i.fyh], xo[i.yh], s);
          s = fma(hzc[i.fz], xo[i.zl], s);
          s = fma(hzo[i.fzh], xo[i.zh], s);
          sum += bv - s;
        }
      }
      a.bc[at(a.dc, p, (y0 >> 1) + J, (z0 >> 1) + K)] = (T)0.5 * sum;
    }
  }
  if (ncta > 1) {  // every CTA has read the base: the last one to finish moves it on
    __syncthreads();
    if (tid == 0) {
      const unsigned done = atomicAdd(a.epoch + 1, 1u);
      if (done == (unsigned)ncta - 1u) {
        a.epoch[1] = 0u;
        a.epoch[0] = base + (unsigned)nhalf;
      }
    }
  }
}

}  // namespace mp
