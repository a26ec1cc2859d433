// Tridiagonal eigensolver ("Solve" in Table 1): divide and conquer on the real symmetric
// tridiagonal T = (d, e), eigenvalues of all of T and eigenvectors of the k lowest.
//
//  * Tearing (Cuppen): at every split m (between rows m-1 and m) with rho = e[m-1]:
//      T = diag(T1 - |rho| e_last e_last^T, T2 - |rho| e_1 e_1^T) + |rho| u u^T,
//      u = e_{m-1} + sign(rho) e_m.
//  * Leaves (<= 16 rows): implicit QL with shifts, one block per leaf.
//  * Merge of two solved children T1' = Q1 D1 Q1^T, T2' = Q2 D2 Q2^T:
//      T' = Q (D + r zz^T) Q^T,  z = [last row of Q1, sign(rho) first row of Q2] / sqrt(2),
//      r = 2|rho|.  The poles (children eigenvalues, each list sorted) are merged by rank;
//      deflation (|r z_i| <= tol, or two poles so close that a Givens rotation zeroing one
//      z-component leaves an off-diagonal <= tol) is tested in parallel, one by one only behind a
//      rotation; the K remaining roots of
//      the secular equation 1 + r sum z_i^2/(delta_i - lambda) = 0 are found one per warp in
//      coordinates shifted to the nearest pole, by a bracketed two-pole rational iteration; z is
//      recomputed from the roots (Gu-Eisenstat) so the eigenvectors u_j = z_i/(delta_i - lambda_j)
//      are numerically orthogonal; the new eigenvectors Q u_j come from two products that use the
//      block structure (columns that live in the top child only, in both, in the bottom only).
//  * Columns are never physically sorted: colmap[a + p] gives the physical column of the p-th
//    smallest eigenvalue of the node starting at a.  At the top merge only the k lowest
//    eigenvectors are formed.
#include <algorithm>
#include <climits>
#include <cmath>
#include <vector>

#include "common.cuh"

namespace gev {

namespace {

constexpr int LEAF = 32;        // rows a leaf kernel holds
// rows of a leaf, at most: the QL chain of 32 rows took 1.0 ms whatever the order, one of 16 rows a quarter, and the
// merge level more costs about 0.15 ms
constexpr int LEAF_ROWS = 16;
constexpr double EPS = 2.220446049250313e-16;

struct Node {
  int a, m, c;       // rows [a, c), split at m
  int K;             // non-deflated count
  int K1, K2, K3;    // top-only / mixed / bottom-only among the non-deflated
  int ndefl;         // deflated count
  int nrot;          // Givens rotations applied
  int Kout;          // eigenvectors to form (roots with final position < kcut)
  double r;          // 2|rho|
  double zn2;        // sum of squared non-deflated z
};

// per-level device arrays carved from the D&C workspace, each of length n (indexed by row range)
struct DcArrays {
  double* dsort;   // merged sorted poles
  double* zs;      // z in sorted order
  int* csrc;       // physical column of each sorted entry
  int* tb;         // bit 1: has rows in the top child, bit 2: in the bottom child
  double* nd_d;    // non-deflated poles (ascending)
  double* nd_z;    // their z
  int* nd_col;     // their physical columns
  int* nd_g;       // gather slot (type order) of each non-deflated entry
  double* df_d;    // deflated eigenvalues (ascending after the sort)
  int* df_col;     // their physical columns
  double* mu;      // root offsets
  int* org;        // root origins (index into nd list)
  double* zp;      // recomputed z
  int* pos_r;      // final position of each root within the node
  int* pos_d;      // final position of each deflated entry
  int* rot_p;      // rotations: column pairs and (c, s)
  int* rot_i;
  double* rot_c;
  double* rot_s;
  int* colmap;     // physical column of each sorted position
  int* colmap2;
  double* dwork;   // torn diagonal
  Node* nodes;     // per-level node descriptors (device)
};

// ------------------------------------------------------------------------------------ tearing --
// dw = d with |e[m-1]| taken off both sides of every leaf boundary m = floor(q n / nleaf)
__global__ void k_tear(int n, int nleaf, const double* d, const double* e, double* dw) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    double v = d[i];
    const int q0 = (int)(((long long)i * nleaf) / n);
    for (int q = max(1, q0 - 1); q <= min(nleaf - 1, q0 + 2); ++q) {
      const int m = (int)(((long long)q * n) / nleaf);
      if (m == i || m == i + 1) v -= fabs(e[m - 1]);
    }
    dw[i] = v;
  }
}

// ------------------------------------------------------------------------------------- leaves --
// 1 / sqrt of q = f^2 + g^2 when q is comfortably inside the range (an integer test of the exponent: an
// FP64 comparison costs as much as a multiplication here); else false and the caller takes hypot
__device__ __forceinline__ bool rsqrt_safe(double q, double& ri) {
  const int e = (__double2hiint(q) >> 20) & 0x7FF;
  if (e < 1023 - 900 || e > 1023 + 900) return false;
  ri = rsqrt(q);
  return true;
}

// Implicit QL on the leaf (rows [a, a+sz)), eigenvectors accumulated in shared memory.  Warp 0 runs the
// scalar recurrence (lane 0; the split search is one ballot) and records each sweep's rotations, warp 1
// (a lane per row) applies the previous sweep's meanwhile: one barrier per sweep.  The recurrence is one
// dependent FP64 chain of about 900 rotations for 32 rows: a rotation is one rsqrt and multiplications
// (hypot and two divisions before, and one thread's split search: 2.4 ms for any matrix of leaves of 32;
// 0.65 ms now).
__global__ void __launch_bounds__(64) k_leaf(int n, int nleaf, const double* dw, const double* e,
                                             double* w, double* Q, long long ldq, int* colmap,
                                             int* status) {
  __shared__ double Z[LEAF][LEAF + 1];
  __shared__ double dd[LEAF], ee[LEAF];
  __shared__ double rc[2][LEAF], rs[2][LEAF];
  __shared__ int s_hi[2], s_nrot[2];  // a sweep's rotations act on columns hi - t, hi - t + 1, t < nrot
  __shared__ int done[2], fail;  // done: by sweep parity, like the rotations
  __shared__ int perm[LEAF];
  const int q = blockIdx.x;
  const int a = (int)(((long long)q * n) / nleaf);
  const int c = (int)(((long long)(q + 1) * n) / nleaf);
  const int sz = c - a;
  const int tid = threadIdx.x, lane = tid & 31;
  for (int i = tid; i < sz; i += blockDim.x) {
    dd[i] = dw[a + i];
    ee[i] = (i + 1 < sz) ? e[a + i] : 0.0;
    for (int j = 0; j < sz; ++j) Z[i][j] = (i == j) ? 1.0 : 0.0;
  }
  if (tid < LEAF) perm[tid] = tid;
  if (tid == 0) { done[0] = done[1] = 0; fail = 0; s_nrot[0] = s_nrot[1] = 0; }
  __syncthreads();
  int l = 0, total = 0, par = 0;  // warp 0's state of the iteration (uniform over the warp)
  while (true) {
    if (tid < 32) {
      int nrot = 0, m = l;
      // the next sweep to perform: the first l with a coupling below it, and the end m of its block
      const bool small = lane + 1 >= sz || fabs(ee[lane]) <= EPS * (fabs(dd[lane]) + fabs(dd[lane + 1 < sz ? lane + 1 : lane]));
      const unsigned cut = __ballot_sync(0xffffffffu, small);
      while (l < sz) {
        m = l + __ffs(cut >> l) - 1;  // (bit sz - 1 is set)
        if (m > l) break;
        ++l;
      }
      bool stop = l >= sz;
      if (!stop && ++total > 30 * sz) {
        stop = true;
        if (lane == 0) fail = 1;
      }
      if (stop) {
        if (lane == 0) done[par] = 1;
      } else if (lane == 0) {
        double g = (dd[l + 1] - dd[l]) / (2.0 * ee[l]);
        double r = hypot(g, 1.0);
        g = dd[m] - dd[l] + ee[l] / (g + copysign(r, g));
        double sn = 1.0, cc = 1.0, p = 0.0;
        bool early = false;
        double ei = ee[m - 1], di = dd[m - 1], dn = dd[m];  // e_i, d_i, d_{i+1}
        for (int i = m - 1; i >= l; --i) {
          const double f = sn * ei, b = cc * ei;
          const double en = i > l ? ee[i - 1] : 0.0, dm = i > l ? dd[i - 1] : 0.0;  // the next step's
          const double qq = fma(f, f, g * g);
          double ri;
          if (rsqrt_safe(qq, ri)) {
            r = qq * ri;
            sn = f * ri;
            cc = g * ri;
          } else {
            r = hypot(f, g);
            if (r == 0.0) { ee[i + 1] = r; dd[i + 1] = dn - p; ee[m] = 0.0; early = true; break; }
            sn = f / r;
            cc = g / r;
          }
          if (i + 1 < m) ee[i + 1] = r;  // (ee[m] is zeroed below)
          g = dn - p;
          const double rr = fma(di - g, sn, 2.0 * cc * b);
          p = sn * rr;
          dd[i + 1] = g + p;
          g = fma(cc, rr, -b);
          rc[par][nrot] = cc;
          rs[par][nrot] = sn;
          ++nrot;
          dn = di;
          di = dm;
          ei = en;
        }
        if (!early) { dd[l] -= p; ee[l] = g; ee[m] = 0.0; }
        s_hi[par] = m - 1;
        s_nrot[par] = nrot;
      }
      __syncwarp();
      if (stop && lane == 0) s_nrot[par] = 0;
    } else if (lane < sz) {
      const int pv = par ^ 1, nr = s_nrot[pv], hi = s_hi[pv];
      if (nr > 0) {
        double z1 = Z[lane][hi + 1];
        for (int t = 0; t < nr; ++t) {
          const int i = hi - t;
          const double zi = Z[lane][i], cs = rc[pv][t], sn = rs[pv][t];
          Z[lane][i + 1] = sn * zi + cs * z1;
          z1 = cs * zi - sn * z1;
        }
        Z[lane][hi - nr + 1] = z1;
      }
    }
    __syncthreads();
    if (done[par]) break;  // (warp 1 has applied the last sweep: done is set in a round without rotations)
    par ^= 1;
  }
  if (tid < 32) {
    if (lane == 0 && fail) atomicCAS(&status[ST_NOCONV], 0, 301);
    if (lane < sz) {  // stable rank of the eigenvalue
      const double v = dd[lane];
      int pos = 0;
      for (int j = 0; j < sz; ++j) {
        const double u = dd[j];
        pos += (u < v || (u == v && j < lane)) ? 1 : 0;
      }
      perm[pos < LEAF ? pos : LEAF - 1] = lane;
    }
  }
  __syncthreads();
  for (int i = tid; i < sz; i += blockDim.x) {
    w[a + i] = dd[perm[i]];
    colmap[a + i] = a + i;
  }
  for (int t = tid; t < sz * sz; t += blockDim.x) {
    const int i = t / sz, j = t % sz;
    Q[(a + j) + (long long)(a + i) * ldq] = Z[j][perm[i]];
  }
}

// ------------------------------------------------------------------------------ merge: prepare --
// exclusive block scan of one 64-bit value per thread (several packed counters); tot: the sum
template <int NTH>
__device__ __forceinline__ unsigned long long block_excl_scan(unsigned long long v, unsigned long long* sm,
                                                               unsigned long long& tot) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long x = v;
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned long long y = __shfl_up_sync(0xffffffffu, x, off);
    if (lane >= off) x += y;
  }
  __syncthreads();  // sm may still be read by the previous scan
  if (lane == 31) sm[wid] = x;
  __syncthreads();
  unsigned long long before = 0, t = 0;
#pragma unroll
  for (int q = 0; q < NTH / 32; ++q) {
    if (q < wid) before += sm[q];
    t += sm[q];
  }
  tot = t;
  return before + x - v;
}

// One block per node: z, rank merge of the two sorted pole lists, deflation, rotations applied to the
// physical columns, sort of the deflated list, gather order by type.
// Deflation looks at one entry after another: an entry with r |z_i| <= tol deflates; else it is tested
// against the last one kept, and where a rotation of the two leaves an off-diagonal <= tol the earlier
// one deflates and the later one, changed, is tested against its successor.  All tests on unchanged
// entries are independent, so they run in parallel and only the entries that follow a rotation are
// tested again, one by one; the lists come from prefix sums.  (As one thread's scan over global memory
// the kernel took 14.8 ms for the top merge at n = 10240 and 2.1 ms at n = 1500: 0.05 ms now at 1500.)
constexpr int PREP_NTH = 512;
__global__ void __launch_bounds__(PREP_NTH) k_merge_prep(int n, int nleaf, int span, Node* nodes, const double* e,
                                                         const double* w, double* Q, long long ldq,
                                                         DcArrays A) {
  Node& nd = nodes[blockIdx.x];
  const int a = (int)(((long long)blockIdx.x * span * n) / nleaf);
  const int m = (int)(((long long)(blockIdx.x * span + span / 2) * n) / nleaf);
  const int c = (int)(((long long)(blockIdx.x + 1) * span * n) / nleaf);
  const int n1 = m - a, nn = c - a;
  const int tid = threadIdx.x;
  constexpr int NTH = PREP_NTH;
  const double rho = e[m - 1];
  const double sg = rho < 0 ? -1.0 : 1.0;
  const double r = 2.0 * fabs(rho);
  const double isq2 = 0.70710678118654752440;
  __shared__ unsigned long long scan_sm[NTH / 32];
  __shared__ double zred[NTH / 32];
  __shared__ int sR, s_next, s_swap;
  // rank merge: child 1 = w[a .. m), child 2 = w[m .. c), both ascending
  for (int i = tid; i < nn; i += NTH) {
    double di;
    int pos, col;
    double zi;
    int tbits;
    if (i < n1) {
      di = w[a + i];
      // number of child-2 entries strictly below di
      int lo = 0, hi = nn - n1;
      while (lo < hi) { int md = (lo + hi) >> 1; if (w[m + md] < di) lo = md + 1; else hi = md; }
      pos = i + lo;
      col = A.colmap[a + i];
      zi = Q[(m - 1) + (long long)col * ldq] * isq2;
      tbits = 1;
    } else {
      const int j = i - n1;
      di = w[m + j];
      int lo = 0, hi = n1;  // child-1 entries <= di
      while (lo < hi) { int md = (lo + hi) >> 1; if (w[a + md] <= di) lo = md + 1; else hi = md; }
      pos = j + lo;
      col = A.colmap[m + j];
      zi = sg * Q[m + (long long)col * ldq] * isq2;
      tbits = 2;
    }
    A.dsort[a + pos] = di;
    A.zs[a + pos] = zi;
    A.csrc[a + pos] = col;
    A.tb[a + pos] = tbits;
  }
  if (tid == 0) { sR = 0; s_next = INT_MAX; }
  __syncthreads();
  const double tol = 8.0 * EPS * fmax(fmax(fabs(A.dsort[a]), fabs(A.dsort[c - 1])), r);
  const int per = (nn + NTH - 1) / NTH, i0 = min(nn, tid * per), i1 = min(nn, i0 + per);
  // the entries that couple (r |z| > tol), in order: index list in A.pos_r; flag 4 in A.tb
  int cnt = 0;
  for (int i = i0; i < i1; ++i) {
    const bool big = !(r * fabs(A.zs[a + i]) <= tol);
    if (big) ++cnt;
    A.pos_d[a + i] = big ? 1 : 0;
  }
  unsigned long long tot;
  int at = (int)block_excl_scan<NTH>((unsigned long long)cnt, scan_sm, tot);
  const int nbig = (int)tot;
  for (int i = i0; i < i1; ++i)
    if (A.pos_d[a + i]) A.pos_r[a + at++] = i;
  __syncthreads();
  // tests of neighbouring kept entries on their original values; rflag (A.org): the pair (q - 1, q) rotates
  for (int q = tid; q < nbig; q += NTH) {
    int fl = 0;
    if (q > 0) {
      const int pj = a + A.pos_r[a + q - 1], ii = a + A.pos_r[a + q];
      const double zp = A.zs[pj], zi = A.zs[ii];
      const double tau = hypot(zp, zi);
      const double cs = zi / tau, sn = zp / tau;
      fl = fabs((A.dsort[ii] - A.dsort[pj]) * cs * sn) <= tol ? 1 : 0;
    }
    A.org[a + q] = fl;
  }
  __syncthreads();
  // the rotations: runs of flagged pairs, by one thread; A.org[q] = 1 in the end: entry q - 1 deflated
  for (int q0 = 1;;) {
    if (tid == 0) s_next = INT_MAX;
    __syncthreads();
    int f = INT_MAX;
    for (int q = q0 + tid; q < nbig; q += NTH)
      if (A.org[a + q]) { f = q; break; }
    if (f != INT_MAX) atomicMin(&s_next, f);
    __syncthreads();
    const int first = s_next;
    __syncthreads();
    if (first == INT_MAX) break;
    if (tid == 0) {
      int q = first, R = sR;
      while (true) {
        const int pj = a + A.pos_r[a + q - 1], ii = a + A.pos_r[a + q];
        const double zp = A.zs[pj], zi = A.zs[ii];
        const double tau = hypot(zp, zi);
        const double cs = zi / tau, sn = zp / tau;
        const double dp = A.dsort[pj], di = A.dsort[ii];
        if (q > first && !(fabs((di - dp) * cs * sn) <= tol)) {
          A.org[a + q] = 0;
          ++q;
          break;
        }
        // rotate the pair so z_prev = 0: prev deflates
        A.org[a + q] = 1;
        A.zs[ii] = tau;
        A.zs[pj] = 0.0;
        A.dsort[pj] = cs * cs * dp + sn * sn * di;
        A.dsort[ii] = sn * sn * dp + cs * cs * di;
        A.rot_p[a + R] = A.csrc[pj];
        A.rot_i[a + R] = A.csrc[ii];
        A.rot_c[a + R] = cs;
        A.rot_s[a + R] = sn;
        ++R;
        const int u = A.tb[pj] | A.tb[ii];
        A.tb[pj] = u;
        A.tb[ii] = u;
        if (++q >= nbig) break;
      }
      sR = R;
      s_next = q;
    }
    __syncthreads();
    q0 = s_next;
    __syncthreads();
  }
  const int R = sR;
  // marks per sorted entry i (A.pos_d): bit 0 couples, bit 1 deflated by a rotation, bit 2 partner of one
  if (R > 0) {
    for (int q = 1 + tid; q < nbig; q += NTH)
      if (A.org[a + q]) {
        atomicOr(&A.pos_d[a + A.pos_r[a + q - 1]], 2);
        atomicOr(&A.pos_d[a + A.pos_r[a + q]], 4);
      }
    __syncthreads();
  }
  // kept entries in order; deflated ones in the order in which the scan meets them (a rotated one when
  // it meets its partner)
  unsigned long long kd = 0;
  double zz = 0.0;
  for (int i = i0; i < i1; ++i) {
    const int f = A.pos_d[a + i];
    if ((f & 3) == 1) kd += 1;
    if (!(f & 1) || (f & 4)) kd += 1ull << 32;
  }
  unsigned long long pre = block_excl_scan<NTH>(kd, scan_sm, tot);
  const int K = (int)(tot & 0xffffffffu), D = (int)(tot >> 32);
  {
    int kp = (int)(pre & 0xffffffffu), dpos = (int)(pre >> 32);
    for (int i = i0; i < i1; ++i) {
      const int f = A.pos_d[a + i];
      if ((f & 3) == 1) {
        const double z = A.zs[a + i];
        A.nd_d[a + kp] = A.dsort[a + i];
        A.nd_z[a + kp] = z;
        A.nd_col[a + kp] = A.csrc[a + i];
        A.nd_g[a + kp] = A.tb[a + i];  // the type bits, replaced by the gather slot below
        zz += z * z;
        ++kp;
      }
      int src = -1;
      if (!(f & 1)) src = i;
      else if (f & 4) {  // the deflated entry is the kept-list predecessor of i
        src = i - 1;
        while (!(A.pos_d[a + src] & 1)) --src;
      }
      if (src >= 0) {
        A.df_d[a + dpos] = A.dsort[a + src];
        A.df_col[a + dpos] = A.csrc[a + src];
        ++dpos;
      }
    }
  }
  for (int off = 16; off > 0; off >>= 1) zz += __shfl_down_sync(0xffffffffu, zz, off);
  if ((tid & 31) == 0) zred[tid >> 5] = zz;
  __syncthreads();
  // stable sort of the deflated list: rotations perturb its order only locally, so transpositions of
  // neighbours, odd and even pairs in turn, end after a few passes
  for (int idle = 0, ph = 0; R > 0 && idle < 2; ph ^= 1) {
    if (tid == 0) s_swap = 0;
    __syncthreads();
    for (int j = ph + 2 * tid; j + 1 < D; j += 2 * NTH) {
      const double d0 = A.df_d[a + j], d1 = A.df_d[a + j + 1];
      if (d0 > d1) {
        const int c0 = A.df_col[a + j];
        A.df_d[a + j] = d1;
        A.df_d[a + j + 1] = d0;
        A.df_col[a + j] = A.df_col[a + j + 1];
        A.df_col[a + j + 1] = c0;
        s_swap = 1;
      }
    }
    __syncthreads();
    idle = s_swap ? 0 : idle + 1;
    __syncthreads();
  }
  // gather order: top-only, mixed, bottom-only (counters packed, 21 bits each)
  {
    const int pk = (K + NTH - 1) / NTH, k0 = min(K, tid * pk), k1 = min(K, k0 + pk);
    unsigned long long t3 = 0;
    for (int i = k0; i < k1; ++i) {
      const int t = A.nd_g[a + i];
      t3 += t == 1 ? 1ull : (t == 3 ? 1ull << 21 : 1ull << 42);
    }
    const unsigned long long p3 = block_excl_scan<NTH>(t3, scan_sm, tot);
    const int K1 = (int)(tot & 0x1fffff), K2 = (int)((tot >> 21) & 0x1fffff), K3 = (int)(tot >> 42);
    int c1 = (int)(p3 & 0x1fffff), c2 = K1 + (int)((p3 >> 21) & 0x1fffff), c3 = K1 + K2 + (int)(p3 >> 42);
    for (int i = k0; i < k1; ++i) {
      const int t = A.nd_g[a + i];
      A.nd_g[a + i] = (t == 1) ? c1++ : (t == 3 ? c2++ : c3++);
    }
    if (tid == 0) {
      double zn2 = 0.0;
      for (int q = 0; q < NTH / 32; ++q) zn2 += zred[q];
      nd.a = a; nd.m = m; nd.c = c;
      nd.K = K; nd.K1 = K1; nd.K2 = K2; nd.K3 = K3; nd.ndefl = D; nd.nrot = R;
      nd.r = r; nd.zn2 = zn2;
      nd.Kout = K;
    }
  }
  // apply the rotations, in order, to the physical columns (rows a .. c-1)
  for (int t = 0; t < R; ++t) {
    const int cp = A.rot_p[a + t], ci = A.rot_i[a + t];
    const double cs = A.rot_c[a + t], sn = A.rot_s[a + t];
    for (int row = a + tid; row < c; row += NTH) {
      const double qp = Q[row + (long long)cp * ldq], qi = Q[row + (long long)ci * ldq];
      Q[row + (long long)cp * ldq] = cs * qp - sn * qi;
      Q[row + (long long)ci * ldq] = sn * qp + cs * qi;
    }
  }
}

// --------------------------------------------------------------------------- merge: secular --
// The secular function and its pieces at mu, by one warp: lane l sums the poles l, l + 32, ...; the
// partial sums are reduced to lane 0 in a fixed order and broadcast, so every lane holds the same bits
// (the root iteration below branches on them identically in all lanes).
__device__ void eval_secular(int K, int j, int o, const double* delta, const double* z, double r,
                             double mu, double& f, double& psi, double& dpsi, double& phi,
                             double& dphi) {
  const int lane = threadIdx.x & 31;
  const double dO = delta[o];
  double a = 0.0, b = 0.0, c = 0.0, e = 0.0;
  for (int i = lane; i < K; i += 32) {
    const double di = (delta[i] - dO) - mu;
    const double zi = z[i];
    const double t = zi * recip(di);
    if (i <= j) { a += zi * t; b += t * t; }
    else { c += zi * t; e += t * t; }
  }
  for (int off = 16; off > 0; off >>= 1) {
    a += __shfl_down_sync(0xffffffffu, a, off);
    b += __shfl_down_sync(0xffffffffu, b, off);
    c += __shfl_down_sync(0xffffffffu, c, off);
    e += __shfl_down_sync(0xffffffffu, e, off);
  }
  psi = __shfl_sync(0xffffffffu, a, 0);
  dpsi = __shfl_sync(0xffffffffu, b, 0);
  phi = __shfl_sync(0xffffffffu, c, 0);
  dphi = __shfl_sync(0xffffffffu, e, 0);
  f = 1.0 + r * (psi + phi);
}

// One warp per root, four to a block (one per scheduler: a warp's FP64 instructions do not wait for another's while
// there are fewer roots than SMs hold); lane 0 writes the result.
__global__ void __launch_bounds__(128) k_secular(Node* nodes, DcArrays A, int* status) {
  const Node nd = nodes[blockIdx.y];
  const int j = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const bool lead = (threadIdx.x & 31) == 0;
  const int K = nd.K;
  if (j >= K) return;  // uniform per warp
  const int a = nd.a;
  const double* delta = A.nd_d + a;
  const double* z = A.nd_z + a;
  const double r = nd.r;
  int o;
  double lo, hi;
  const bool last = (j == K - 1);
  if (!last) {
    const double gap = delta[j + 1] - delta[j];
    const double mid = 0.5 * gap;
    double f, psi, dpsi, phi, dphi;
    eval_secular(K, j, j, delta, z, r, mid, f, psi, dpsi, phi, dphi);
    if (f >= 0.0) { o = j; lo = 0.0; hi = mid; }
    else { o = j + 1; lo = -mid; hi = 0.0; }
  } else {
    o = j;
    lo = 0.0;
    hi = r * nd.zn2;
  }
  const double dO = delta[o];
  const double D1b = delta[j] - dO;                       // left pole of the interval (shifted)
  const double D2b = last ? 0.0 : delta[j + 1] - dO;      // right pole (unused for the last root)
  double mu = 0.5 * (lo + hi);
  bool conv = false;
  for (int it = 0; it < 200; ++it) {
    double f, psi, dpsi, phi, dphi;
    eval_secular(K, j, o, delta, z, r, mu, f, psi, dpsi, phi, dphi);
    if (f == 0.0) { conv = true; break; }
    if (f < 0.0) lo = mu; else hi = mu;
    const double errb = 8.0 * EPS * (double)(K + 2) * (1.0 + r * (fabs(psi) + fabs(phi)));
    if (fabs(f) <= errb) { conv = true; break; }
    if (hi - lo <= 4.0 * EPS * fmax(fabs(lo), fabs(hi))) { conv = true; break; }
    // two-pole rational model g(x) = a + q/(D1 - eta) + Q/(D2 - eta), eta = x - mu
    double eta;
    const double D1 = D1b - mu;
    const double q = r * dpsi * D1 * D1;
    if (!last) {
      const double D2 = D2b - mu;
      const double Qc = r * dphi * D2 * D2;
      const double aa = f - q / D1 - Qc / D2;
      const double c0 = D1 * D2 * f;
      const double b0 = aa * (D1 + D2) + q + Qc;
      if (aa == 0.0) {
        eta = c0 / b0;
      } else {
        double disc = b0 * b0 - 4.0 * aa * c0;
        disc = disc > 0.0 ? sqrt(disc) : 0.0;
        double e1, e2;
        if (b0 >= 0.0) { e1 = (b0 + disc) / (2.0 * aa); e2 = 2.0 * c0 / (b0 + disc); }
        else { e1 = (b0 - disc) / (2.0 * aa); e2 = 2.0 * c0 / (b0 - disc); }
        const bool in1 = (mu + e1 > lo) && (mu + e1 < hi);
        const bool in2 = (mu + e2 > lo) && (mu + e2 < hi);
        eta = in2 ? e2 : (in1 ? e1 : 0.5 * (lo + hi) - mu);
      }
    } else {
      const double aa = f - q / D1;
      eta = (aa != 0.0) ? D1 + q / aa : 0.5 * (lo + hi) - mu;
    }
    double mnew = mu + eta;
    const bool ok = last ? (mnew > lo && mnew <= hi) : (mnew > lo && mnew < hi);
    if (!ok || !(mnew == mnew)) mnew = 0.5 * (lo + hi);
    if (fabs(mnew - mu) <= 2.0 * EPS * fabs(mnew)) { mu = mnew; conv = true; break; }
    mu = mnew;
  }
  if (!lead) return;
  if (!conv) atomicCAS(&status[ST_NOCONV], 0, 302);
  A.mu[a + j] = mu;
  A.org[a + j] = o;
}

// Gu-Eisenstat: z'_i^2 = prod_j (lambda_j - delta_i) / (r prod_{j != i} (delta_j - delta_i)).
// One warp per entry: the lanes take the factors j = lane, lane + 32, ..., two factors to a division (an
// FP64 division costs about ten multiplications), and their products are multiplied in a fixed order.
// By interlacing every factor is in (0, 1), so no partial product is smaller than the whole; the products
// of two differences stay in range while the poles' spread does (pair, else one division per factor).
// (One thread per entry before, a chain of divisions: 9.3 ms for all levels at n = 10240, 2.7 ms now.)
__global__ void __launch_bounds__(256) k_zprime(Node* nodes, DcArrays A) {
  const Node nd = nodes[blockIdx.y];
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int K = nd.K;
  if (i >= K) return;  // uniform per warp
  const int a = nd.a;
  const double* delta = A.nd_d + a;
  const double* mu = A.mu + a;
  const int* org = A.org + a;
  const double di = delta[i];
  auto lam_minus = [&](int j) { return (delta[org[j]] - di) + mu[j]; };
  auto den = [&](int j) { return delta[j < i ? j : j + 1] - di; };
  const double spread = fmax(delta[K - 1] - delta[0], nd.r * nd.zn2);
  const bool pair = spread > 1e-100 && spread < 1e100;
  double prod = 1.0;
  int j = lane;
  if (pair) {
    for (; j + 32 < K - 1; j += 64) {
      const double num = lam_minus(j) * lam_minus(j + 32), dd = den(j) * den(j + 32);
      prod *= num / dd;
    }
  }
  for (; j < K - 1; j += 32) prod *= lam_minus(j) / den(j);
  for (int off = 16; off > 0; off >>= 1) prod *= __shfl_down_sync(0xffffffffu, prod, off);
  if (lane == 0) {
    prod *= lam_minus(K - 1) / nd.r;
    A.zp[a + i] = copysign(sqrt(fabs(prod)), A.nd_z[a + i]);
  }
}

// Final positions of roots and deflated entries within each node; eigenvalues in sorted order.
__global__ void k_positions(Node* nodes, DcArrays A) {
  Node& nd = nodes[blockIdx.y];
  const int a = nd.a, K = nd.K, D = nd.ndefl;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < K + D; t += gridDim.x * blockDim.x) {
    if (t < K) {
      const double lam = A.nd_d[a + A.org[a + t]] + A.mu[a + t];
      int lo = 0, hi = D;
      while (lo < hi) { int md = (lo + hi) >> 1; if (A.df_d[a + md] < lam) lo = md + 1; else hi = md; }
      A.pos_r[a + t] = t + lo;
    } else {
      const int u = t - K;
      const double dv = A.df_d[a + u];
      int lo = 0, hi = K;
      while (lo < hi) {
        int md = (lo + hi) >> 1;
        const double lam = A.nd_d[a + A.org[a + md]] + A.mu[a + md];
        if (lam <= dv) lo = md + 1; else hi = md;
      }
      A.pos_d[a + u] = u + lo;
    }
  }
}

// The roots of the top merge whose position is below kcut are a prefix of their list (positions increase): Kout, by
// bisection.  The deflation count goes to the status words.
__global__ void k_count_out(Node* nodes, DcArrays A, int kcut, int* status) {
  Node& nd = nodes[0];
  if (threadIdx.x > 0) return;
  const int* pos = A.pos_r + nd.a;
  int lo = 0, hi = nd.K;
  while (lo < hi) {
    const int md = (lo + hi) >> 1;
    if (pos[md] < kcut) lo = md + 1;
    else hi = md;
  }
  nd.Kout = lo;
  status[ST_DEFLATED] = nd.ndefl;
}

// U (gather order rows x Kout, ld ldu) column j: u_i = z'_i/(delta_i - lambda_j), normalised.
__global__ void k_vectors(Node* nodes, DcArrays A, double* U, long long ldu) {
  const Node nd = nodes[blockIdx.y];
  const int j = blockIdx.x;
  if (j >= nd.Kout) return;
  const int a = nd.a, K = nd.K;
  const double* delta = A.nd_d + a;
  const double dO = delta[A.org[a + j]];
  const double mu = A.mu[a + j];
  double* col = U + (long long)(a + j) * ldu;  // rows 0 .. K-1 of column a + j
  double ss = 0.0;
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    const double v = A.zp[a + i] * recip((delta[i] - dO) - mu);
    col[A.nd_g[a + i]] = v;
    ss += v * v;
  }
  __shared__ double red[32];
  for (int off = 16; off > 0; off >>= 1) ss += __shfl_down_sync(0xffffffffu, ss, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += red[q];
    red[0] = 1.0 / sqrt(t);
  }
  __syncthreads();
  const double inv = red[0];
  for (int i = threadIdx.x; i < K; i += blockDim.x) col[i] *= inv;
}

// Qg[:, a + g] = Q[:, nd_col] (rows a .. c-1) in gather order; deflated columns go straight to
// Qout[:, a + K + u].
__global__ void k_gather(Node* nodes, DcArrays A, const double* Q, long long ldq, double* Qg,
                         double* Qout) {
  const Node nd = nodes[blockIdx.y];
  const int a = nd.a, c = nd.c, nn = c - a;
  const int t = blockIdx.x;
  if (t < nd.K) {
    const int src = A.nd_col[a + t];
    const int g = A.nd_g[a + t];
    for (int i = threadIdx.x; i < nn; i += blockDim.x)
      Qg[(a + i) + (long long)(a + g) * ldq] = Q[(a + i) + (long long)src * ldq];
  } else if (t < nd.K + nd.ndefl) {
    const int u = t - nd.K;
    const int src = A.df_col[a + u];
    for (int i = threadIdx.x; i < nn; i += blockDim.x)
      Qout[(a + i) + (long long)(a + nd.K + u) * ldq] = Q[(a + i) + (long long)src * ldq];
  }
}

// Sorted eigenvalues and the column map of the merged node.
__global__ void k_finalize(Node* nodes, DcArrays A, double* w) {
  const Node nd = nodes[blockIdx.y];
  const int a = nd.a, K = nd.K, D = nd.ndefl;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < K + D; t += gridDim.x * blockDim.x) {
    if (t < K) {
      const int p = A.pos_r[a + t];
      w[a + p] = A.nd_d[a + A.org[a + t]] + A.mu[a + t];
      A.colmap2[a + p] = a + t;
    } else {
      const int u = t - K;
      const int p = A.pos_d[a + u];
      w[a + p] = A.df_d[a + u];
      A.colmap2[a + p] = a + K + u;
    }
  }
}

// The eigenvector products of all nodes of a level in one launch, for levels of short nodes: top rows
// Qb(a.., :) = Qg(a.., top-only and mixed) U(0 .., :), bottom rows Qb(m.., :) = Qg(m.., mixed and
// bottom-only) U(K1 .., :).  blockIdx.z = 2 node + half, 16 x 16 outputs per block, one per thread; R: the
// type of the products and sums (FP32 in the mixed form).  On the FP64 pipe (1.7 multiply-adds per SM
// per cycle) a level of nodes of s rows takes about n s^2 / 2 of them, spread over all SMs, where the
// tensor-core engine takes a split and a product launch (about 35 us) for each half of each node.  The whole
// divide and conquer (with the scans above): n = 256 4.2 -> 1.6 ms, n = 1500 12.8 -> 3.5, n = 10240 113.7 -> 53.0.
constexpr int MT = 16, MK = 32;
template <class R>
__global__ void __launch_bounds__(MT * MT) k_merge_products(const Node* nodes, const double* Qg, const double* U,
                                                            long long ldq, double* Qb) {
  const Node& nd = nodes[blockIdx.z >> 1];
  const int half = blockIdx.z & 1;
  const int a = nd.a, r0 = half ? nd.m : a, nrow = half ? nd.c - nd.m : nd.m - a, Kout = nd.Kout;
  const int i0 = blockIdx.x * MT, j0 = blockIdx.y * MT;
  if (i0 >= nrow || j0 >= Kout) return;
  const int k0 = half ? nd.K1 : 0, KK = half ? nd.K2 + nd.K3 : nd.K1 + nd.K2;
  __shared__ R As[MK][MT + 1], Bs[MT][MK + 1];
  const int tid = threadIdx.x, ti = tid % MT, tj = tid / MT;
  const double* Aq = Qg + r0 + (long long)(a + k0) * ldq;
  const double* Bq = U + (long long)a * ldq + k0;
  R acc0 = 0, acc1 = 0;
  for (int kb = 0; kb < KK; kb += MK) {
    for (int t = tid; t < MT * MK; t += MT * MT) {
      const int i = t % MT, k = t / MT;
      As[k][i] = (i0 + i < nrow && kb + k < KK) ? (R)Aq[i0 + i + (long long)(kb + k) * ldq] : (R)0;
      const int kk = t % MK, j = t / MK;
      Bs[j][kk] = (j0 + j < Kout && kb + kk < KK) ? (R)Bq[kb + kk + (long long)(j0 + j) * ldq] : (R)0;
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < MK; k += 2) {
      acc0 += As[k][ti] * Bs[tj][k];
      acc1 += As[k + 1][ti] * Bs[tj][k + 1];
    }
    __syncthreads();
  }
  if (i0 + ti < nrow && j0 + tj < Kout) Qb[r0 + i0 + ti + (long long)(a + j0 + tj) * ldq] = (double)(acc0 + acc1);
}

// Z[:, p] = Q[:, colmap[p]] for p < k (rows 0 .. n-1).
__global__ void k_output(int n, int k, const double* Q, long long ldq, const int* colmap, double* Z,
                         long long ldz) {
  const int p = blockIdx.x;
  if (p >= k) return;
  const int src = colmap[p];
  for (int i = threadIdx.x; i < n; i += blockDim.x) Z[i + (long long)p * ldz] = Q[i + (long long)src * ldq];
}

}  // namespace

int stedc(Sys& s, const double* d, const double* e, int k, double* w, double* Z, int ldz, int* deflated) {
  const int n = s.n;
  cudaStream_t st = s.stream;
  // carve the workspace
  char* p = (char*)s.dcws;
  auto take = [&](size_t bytes) {
    char* r = p;
    p += (bytes + 255) & ~(size_t)255;
    return (void*)r;
  };
  DcArrays A;
  const size_t nd8 = sizeof(double) * (size_t)n, ni4 = sizeof(int) * (size_t)n;
  A.dsort = (double*)take(nd8); A.zs = (double*)take(nd8); A.csrc = (int*)take(ni4); A.tb = (int*)take(ni4);
  A.nd_d = (double*)take(nd8); A.nd_z = (double*)take(nd8); A.nd_col = (int*)take(ni4); A.nd_g = (int*)take(ni4);
  A.df_d = (double*)take(nd8); A.df_col = (int*)take(ni4); A.mu = (double*)take(nd8); A.org = (int*)take(ni4);
  A.zp = (double*)take(nd8); A.pos_r = (int*)take(ni4); A.pos_d = (int*)take(ni4);
  A.rot_p = (int*)take(ni4); A.rot_i = (int*)take(ni4); A.rot_c = (double*)take(nd8); A.rot_s = (double*)take(nd8);
  A.colmap = (int*)take(ni4); A.colmap2 = (int*)take(ni4); A.dwork = (double*)take(nd8);
  A.nodes = (Node*)take(sizeof(Node) * (size_t)(n / 2 + 2));
  if ((size_t)(p - (char*)s.dcws) > s.dcws_bytes) return GEV_ERR_OOM;
  // every list entry is a valid index from the start: where the input holds NaN, ranks collide and entries stay
  // unwritten
  GEV_CUDA_TRY(cudaMemsetAsync(s.dcws, 0, (size_t)(p - (char*)s.dcws), st));

  double* Qa = s.Q;
  double* Qb = s.Q2;
  double* Qg = (double*)s.W1;
  double* U = (double*)s.Yk;  // s.A keeps the FP64 standard matrix (mixed-form refinement)
  const long long ldq = n;

  // Every column of a node must be zero outside the node's rows (block-diagonal eigenvector
  // matrices): deflated columns are copied over the whole node range and Givens rotations mix full
  // columns.  Both buffers are cleared here, so rows a level never writes stay zero.
  GEV_CUDA_TRY(cudaMemsetAsync(Qa, 0, sizeof(double) * (size_t)n * n, st));
  GEV_CUDA_TRY(cudaMemsetAsync(Qb, 0, sizeof(double) * (size_t)n * n, st));
  int nleaf = 1;
  while ((n + nleaf - 1) / nleaf > LEAF_ROWS) nleaf *= 2;
  const unsigned eb = cdiv(n, 256) < 1024u ? cdiv(n, 256) : 1024u;
  GEV_CUDA_TRY(cudaMemsetAsync(&s.status[ST_DEFLATED], 0, sizeof(int), st));
  GEV_COUNT(s);
  k_tear<<<eb, 256, 0, st>>>(n, nleaf, d, e, A.dwork);
  GEV_COUNT(s);
  k_leaf<<<nleaf, 64, 0, st>>>(n, nleaf, A.dwork, e, w, Qa, ldq, A.colmap, s.status);
  GEV_TRY(last_error());

  // Levels whose nodes have at most kBatch rows run their products in one launch with everything read
  // from the node descriptors on the device, so the host does not wait for them: n s^2 / 2 multiply-adds on the
  // FP64 pipe (4.5e11 per second over the chip) against 2 n / s products of about 35 us: equal at s about 390
  // for any n.
  constexpr int kBatch = 384;
  std::vector<Node> hn;
  for (int span = 2; span <= nleaf; span *= 2) {
    const int nnodes = nleaf / span;
    const bool top = (span == nleaf);
    const int smax = (int)std::min<long long>(n, ((long long)span * n) / nleaf + 1);  // rows of a node, at most
    const bool batch = smax <= kBatch;
    GEV_COUNT(s);
    k_merge_prep<<<nnodes, PREP_NTH, 0, st>>>(n, nleaf, span, A.nodes, e, w, Qa, ldq, A);
    GEV_TRY(last_error());
    GEV_COUNT(s);
    k_secular<<<dim3(cdiv(smax, 4), nnodes), 128, 0, st>>>(A.nodes, A, s.status);
    GEV_COUNT(s);
    k_zprime<<<dim3(cdiv(smax, 8), nnodes), 256, 0, st>>>(A.nodes, A);
    const int kcut = top ? k : 0x7fffffff;
    GEV_COUNT(s);
    k_positions<<<dim3(cdiv(smax, 256), nnodes), 256, 0, st>>>(A.nodes, A);
    if (top) {
      GEV_COUNT(s);
      k_count_out<<<1, 32, 0, st>>>(A.nodes, A, kcut, s.status);
    }
    GEV_TRY(last_error());
    GEV_COUNT(s);
    k_vectors<<<dim3(smax, nnodes), 256, 0, st>>>(A.nodes, A, U, ldq);
    GEV_COUNT(s);
    k_gather<<<dim3(smax, nnodes), 256, 0, st>>>(A.nodes, A, Qa, ldq, Qg, Qb);
    GEV_TRY(last_error());
    // eigenvector update: top rows use the top-only and mixed columns, bottom rows the mixed and
    // bottom-only ones
    if (batch) {
      const dim3 grid(cdiv((smax + 1) / 2 + 1, MT), cdiv(smax, MT), 2 * nnodes);
      GEV_COUNT(s);
      if (s.dc_lowp) k_merge_products<float><<<grid, MT * MT, 0, st>>>(A.nodes, Qg, U, ldq, Qb);
      else k_merge_products<double><<<grid, MT * MT, 0, st>>>(A.nodes, Qg, U, ldq, Qb);
      GEV_TRY(last_error());
    } else {
      hn.resize(nnodes);
      GEV_CUDA_TRY(cudaMemcpyAsync(hn.data(), A.nodes, sizeof(Node) * nnodes, cudaMemcpyDeviceToHost, st));
      GEV_CUDA_TRY(cudaStreamSynchronize(st));
    }
    for (int q = 0; !batch && q < nnodes; ++q) {
      const Node& x = hn[q];
      if (x.Kout == 0) continue;
      const int n1 = x.m - x.a, n2 = x.c - x.m;
      const double* Ub = U + (long long)x.a * ldq;  // column a, rows 0 .. K-1 (gather order)
      if (x.K1 + x.K2 > 0)
      {
        GemmP<double> g = gp<double>(n1, x.Kout, x.K1 + x.K2, 0, 0, 1.0, Qg + x.a + (long long)x.a * ldq, ldq,
                                     Ub, ldq, 0.0, Qb + x.a + (long long)x.a * ldq, ldq);
        g.lowp = s.dc_lowp;
        gemm(s, g);
      }
      else
        GEV_CUDA_TRY(cudaMemset2DAsync(Qb + x.a + (long long)x.a * ldq, ldq * 8, 0, n1 * 8, x.Kout, st));
      if (x.K2 + x.K3 > 0)
      {
        GemmP<double> g = gp<double>(n2, x.Kout, x.K2 + x.K3, 0, 0, 1.0, Qg + x.m + (long long)(x.a + x.K1) * ldq,
                                     ldq, Ub + x.K1, ldq, 0.0, Qb + x.m + (long long)x.a * ldq, ldq);
        g.lowp = s.dc_lowp;
        gemm(s, g);
      }
      else
        GEV_CUDA_TRY(cudaMemset2DAsync(Qb + x.m + (long long)x.a * ldq, ldq * 8, 0, n2 * 8, x.Kout, st));
    }
    GEV_COUNT(s);
    k_finalize<<<dim3(cdiv(smax, 256), nnodes), 256, 0, st>>>(A.nodes, A, w);
    GEV_TRY(last_error());
    std::swap(A.colmap, A.colmap2);
    std::swap(Qa, Qb);
  }
  // the k lowest eigenvectors
  GEV_COUNT(s);
  k_output<<<k, 256, 0, st>>>(n, k, Qa, ldq, A.colmap, Z, ldz);
  GEV_TRY(last_error());
  if (deflated) {
    GEV_CUDA_TRY(cudaMemcpyAsync(deflated, &s.status[ST_DEFLATED], sizeof(int), cudaMemcpyDeviceToHost, st));
    GEV_CUDA_TRY(cudaStreamSynchronize(st));
  }
  return 0;
}

}  // namespace gev
