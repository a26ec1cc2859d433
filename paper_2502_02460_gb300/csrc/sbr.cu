// Stage 1 of the two-stage tridiagonalisation ("ELPA2", section "Usability and Tutorials"):
// full Hermitian A -> band B of width b, A = Q1 B Q1^H, and the matching back-transform Y = Q1 Z.
//
// For each panel (columns j0..j0+b-1, rows r0 = j0+b .. n-1):
//   1. Householder QR of the m x b panel (m = n - r0) in ONE kernel: the panel rows are spread over the
//      blocks and stay in shared memory; each column needs one barrier (the norm and the reflector's
//      inner products together, which also give the column of the compact-WY factor T).  Long panels: a
//      cooperative grid over all SMs, whose barrier gives up after a bounded wait; short ones: one cluster
//      of 16 blocks and its hardware barrier, which has no limit and needs none (all blocks of a cluster
//      run, and none leaves before the last column).  Q = H_0 ... H_{b-1} = I - Y T Y^H, T upper triangular.
//   2. Two-sided update of the trailing block A22 <- Q^H A22 Q by GEMMs:
//        W = A22 Y T,  U = T^H (Y^H W),  V = W - Y U / 2,  A22 -= [Y V] [V Y]^H (lower, one
//        rank-2b product), mirror.
// Y is kept explicitly (unit diagonal, zeros above) in the handle's V1 at the panel's position and
// T in T1, for the back-transform  Y_out = Q1 Z = Q_0 (Q_1 (... Q_last Z)).
#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "coop.cuh"
#include "int_sums.cuh"

namespace gev {

namespace {

// threads of a panel block: four (b = 16: eight) per column.  All four schedulers have a warp then, and the sums
// over a column's threads, a chain of FP64 additions in one warp, stay short.
template <int B> constexpr int panel_nt() { return B == 64 ? 256 : 128; }

template <class T> struct PanelArgs {
  int m, R, use_smem, t_smem;
  T* P;
  long long ldp;
  T* Y;     // the reflectors: in V1 and, for the trailing update, in up to three panel buffers
  T* Y1;
  T* Y2;
  T* Y3;
  long long ldy;
  T* Tm;
  double* nrm_part;
  T* w_part;
  T* prow;
  int* count;  // arrivals, since the reduction began; base: before this launch
  int base;
  int* status;
  int* abort_flag;
};

// Householder QR of the m x B panel, one grid barrier per column.  Before the barrier every block sums,
// over its rows below the pivot, u_j = sum_r conj(x_r) P(r, j) with the current column x (j > c: the columns
// to update; j < c: the reflectors before, for T; j = c: ||x||^2), and the block holding the pivot row
// publishes that row.  After the barrier each block adds the block sums in a fixed order, forms the
// reflector (beta, tau, scale: v_c = 1, v_r = scale x_r) and recovers the inner products exactly as
//   w_j = v^H P(:, j) = P(c, j) + conj(scale) u_j,     s_j = Y(:, j)^H v = conj(sc_j) (conj(P(c, j)) + scale conj(u_j)).
// The stored columns stay unscaled (their scales sc_j are applied when Y is written), so a column costs
// one pass over the block's rows before the barrier and one after it.
//
// The column is a chain of latencies, not of work (m B multiply-adds over all SMs: 0.3 - 2 us): the
// partial sums and the barrier's flag travel through L2 once each, all partial sums a thread adds are
// loaded together (20 or 40 at a time), the reflector is one reciprocal root and one reciprocal, and the two warps
// that need its inner products compute it themselves.  Per panel, averages over a reduction: n = 1500, b = 32
// 275 us at first, 127 now (in a cluster); n = 10240, b = 64 782 -> 410; complex n = 509, b = 32 440 -> 270 (grid form).
// The partial-sum buffers alternate with the column's parity: a block may start column c + 1 while a
// slower one still reads column c's sums, but column c + 2 waits for everyone at barrier c + 1.
//
// CL > 0: the whole panel in one cluster of CL blocks.  A block then sends its sums (and the pivot row) to every block's
// shared memory, and the grid barrier becomes the cluster's: no release through L2 (about 1000 cycles), no polls, no
// partial sums from L2, CL of them instead of the grid's 50 to 150.  A block's shared memory may only be written once it
// is known to run, so one cluster barrier stands before the first column; its arrivals overlap the load of the rows.
template <class T, int B, int CL>
__global__ void __launch_bounds__(panel_nt<B>()) k_panel_qr(PanelArgs<T> a) {
  constexpr int NT = panel_nt<B>(), NG = NT / B;
  constexpr bool LOW = sizeof(typename real_of<T>::type) == 4;  // FP32 data: norms in FP64
  constexpr int NLD = sizeof(T) == 16 ? 20 : 40;                // partial sums in flight per thread
  extern __shared__ __align__(16) unsigned char smraw[];
  const int blk = blockIdx.x, tid = threadIdx.x, G = gridDim.x, m = a.m;
  const int lo = blk * a.R, hi = min(m, lo + a.R), rows = max(0, hi - lo);
  const long long lds = a.R | 1;
  if constexpr (CL > 0) asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
  T* red2 = reinterpret_cast<T*>(smraw);  // NT
  T* wv = red2 + NT;                      // B: factors of the pivot row, then of s_j
  T* w2 = wv + B;                         // B: factors of the rows below
  T* sc = w2 + B;                         // B: scales of the reflectors
  double* redn = reinterpret_cast<double*>(sc + B);  // NT / 32 + NG
  T* Ts = reinterpret_cast<T*>(redn + NT / 32 + NG); // B x B when t_smem
  T* cw = Ts + (a.t_smem ? B * B : 0);               // cluster: 2 x CL x B sums, 2 x B pivot row, 2 x CL norms
  T* cp = cw + 2 * CL * B;
  double* cn = reinterpret_cast<double*>(cp + (CL ? 2 * B : 0));
  T* sm = reinterpret_cast<T*>(cn + 2 * CL);         // the block's rows when use_smem
  __shared__ T sh_beta;
  __shared__ int s_ok;
  T* Tw = a.t_smem ? Ts : a.Tm;
  T* base = a.use_smem ? sm : a.P + lo;
  const long long ld = a.use_smem ? lds : a.ldp;
  if (a.use_smem)
    for (int idx = tid; idx < rows * B; idx += NT) {
      const int r = idx % rows, c = idx / rows;
      sm[r + c * lds] = a.P[(lo + r) + c * a.ldp];
    }
  __syncthreads();
  if constexpr (CL > 0) asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");  // every block has started
  const int jj = tid % B, grp = tid / B;
  const int ncol = min(B, m);
  // column c of T from the inner products in wv: T(0:c, c) = -tau T(0:c, 0:c) s, T(c, c) = tau; B threads
  auto t_column = [&](int c) {
    const int i = tid - (NT - B);
    const T tau = wv[c];
    T val = zero_<T>();
    if (i < c) {
      T acc = zero_<T>(), acc1 = zero_<T>();
      int l = i;
      for (; l + 1 < c; l += 2) {
        mac(acc, Tw[i + l * B], wv[l]);
        mac(acc1, Tw[i + (l + 1) * B], wv[l + 1]);
      }
      if (l < c) mac(acc, Tw[i + l * B], wv[l]);
      val = -(tau * (acc + acc1));
    } else if (i == c) {
      val = tau;
    }
    Tw[i + c * B] = val;
  };

  for (int c = 0; c < ncol; ++c) {
    const int par = c & 1;
    double* np_ = a.nrm_part + (size_t)par * 4096;
    T* wp_ = a.w_part + (size_t)par * 4096 * B;
    T* pr_ = a.prow + (size_t)par * B;
    // ---- A: partial sums over this block's rows strictly below the pivot
    {
      T acc = zero_<T>();
      double ss = 0.0;
      for (int r = max(0, c + 1 - lo) + grp; r < rows; r += NG) {
        const T x = base[r + c * ld];
        cmac(acc, x, base[r + jj * ld]);
        if (LOW && jj == c) ss += abs2_(x);
      }
      red2[tid] = acc;
      if (LOW && jj == c) redn[NT / 32 + grp] = ss;
    }
    __syncthreads();
    if constexpr (CL > 0) {
      // group g sends to the blocks g, g + NG, ..
      T sum = red2[jj];
#pragma unroll
      for (int g = 1; g < NG; ++g) sum += red2[g * B + jj];
      const bool piv = lo <= c && c < hi;
      const T pv = piv ? base[(c - lo) + jj * ld] : zero_<T>();
      double nn = 0.0;
      if (LOW && jj == c)
        for (int g = 0; g < NG; ++g) nn += redn[NT / 32 + g];
      for (int q = grp; q < CL; q += NG) {
        st_peer(peer_addr(smem_u32(&cw[(par * CL + blk) * B + jj]), q), sum);
        if (piv) st_peer(peer_addr(smem_u32(&cp[par * B + jj]), q), pv);
        if (LOW && jj == c) st_peer(peer_addr(smem_u32(&cn[par * CL + blk]), q), nn);
      }
      __syncwarp();
      asm volatile("barrier.cluster.arrive.release.aligned;\n" ::: "memory");
      // column c - 1 of T, while the others arrive
      if (blk == 0 && c > 0 && tid >= NT - B) t_column(c - 1);
      __syncwarp();
      asm volatile("barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
    } else {
      if (tid < B) {
        T sum = red2[tid];
#pragma unroll
        for (int g = 1; g < NG; ++g) sum += red2[g * B + tid];
        stcg_(&wp_[(long long)blk * B + tid], sum);
        if (lo <= c && c < hi) stcg_(&pr_[tid], base[(c - lo) + tid * ld]);  // the pivot row
        if (LOW && tid == c) {
          double s = 0.0;
          for (int g = 0; g < NG; ++g) s += redn[NT / 32 + g];
          __stcg(&np_[blk], s);
        }
      }
      __syncthreads();
      // column c - 1 of T, while the others arrive (its inner products are in wv until the barrier)
      if (blk == 0 && c > 0 && tid >= NT - B) t_column(c - 1);
      if (tid == 0) {
        asm volatile("red.release.gpu.global.add.s32 [%0], 1;\n" ::"l"(a.count) : "memory");
        const int target = a.base + (c + 1) * G;
        int ok = 1;
        if (ld_acquire(a.count) < target) {
          volatile int* vab = a.abort_flag;
          const long long lim = spin_limit(a.status);
          long long it = 0;
          while (ld_acquire(a.count) < target) {
            if (*vab) { ok = 0; break; }
            if (++it > lim) {
              atomicCAS(&a.status[ST_TIMEOUT], 0, 101);
              atomicExch(a.abort_flag, 1);
              ok = 0;
              break;
            }
            if (it > 64) __nanosleep(32);
          }
        }
        s_ok = ok;
      }
      __syncthreads();
      if (!s_ok) return;
    }
    // ---- B: the block sums, added by NG threads per column
    T pc = zero_<T>(), alpha = zero_<T>();
    if (tid < B) {
      pc = CL ? cp[par * B + tid] : ldcg_(&pr_[tid]);
      alpha = CL ? cp[par * B + c] : ldcg_(&pr_[c]);
    }
    {
      T part = zero_<T>();
      if constexpr (CL > 0) {
#pragma unroll
        for (int q = 0; q < CL; q += NG)
          if (q + grp < CL) part += cw[(par * CL + q + grp) * B + jj];
      }
      for (int q0 = grp; CL == 0 && q0 < G; q0 += NLD * NG) {
        T v[NLD];
#pragma unroll
        for (int u = 0; u < NLD; ++u) {
          const int q = q0 + u * NG;
          v[u] = q < G ? ldcg_(&wp_[(long long)q * B + jj]) : zero_<T>();
        }
        part += sum_block(v);
      }
      red2[tid] = part;
      if (LOW) {
        double x = 0.0;
        for (int q = tid; q < G; q += NT) x += CL ? cn[par * CL + q] : __ldcg(&np_[q]);
        for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
        if ((tid & 31) == 0) redn[tid >> 5] = x;
      }
    }
    __syncthreads();
    if (tid < B) {
      T sum = red2[tid];
      double xn;
      if (LOW) {
        xn = 0.0;
        for (int g = 0; g < NT / 32; ++g) xn += redn[g];
      } else {
        xn = (double)re_(red2[c]);
      }
#pragma unroll
      for (int g = 1; g < NG; ++g) {
        sum += red2[g * B + tid];
        if (!LOW && B > 32) xn += re_(red2[g * B + c]);
      }
      if (!LOW && B <= 32) xn = __shfl_sync(B == 32 ? 0xffffffffu : 0xffffu, (double)re_(sum), c);
      T tau = zero_<T>(), beta = alpha, scale = zero_<T>();
      if (!(xn == 0.0 && im_(alpha) == 0)) {
        if constexpr (LOW) {  // the norm in FP64; the rest as the data
          const float nrm = norm_low((double)abs2_(alpha) + xn);
          beta = from_re<T>(re_(alpha) >= 0.f ? -nrm : nrm);
          tau = div_(beta - alpha, beta);
          scale = div_(from_re<T>(1.0), alpha - beta);
        } else {
          house(alpha, xn, tau, beta, scale);
        }
      }
      if (tid > c) {
        const T w = conj_(tau) * (pc + conj_(scale) * sum);
        wv[tid] = w;
        w2[tid] = scale * w;
      } else if (tid < c) {
        wv[tid] = conj_(sc[tid]) * (conj_(pc) + scale * conj_(sum));
      } else {
        wv[tid] = tau;
        sh_beta = beta;
      }
      // (sc[c] is read by no other thread before the barrier below)
      if (tid == c) sc[c] = scale;
    }
    __syncthreads();
    // ---- C: apply H^H to the remaining columns
    if (jj > c) {
      const T w = w2[jj];
      for (int r = max(0, c + 1 - lo) + grp; r < rows; r += NG) nmac(base[r + jj * ld], base[r + c * ld], w);
    }
    if (lo <= c && c < hi && tid < B && tid >= c) {
      if (tid > c) base[(c - lo) + tid * ld] -= wv[tid];
      else base[(c - lo) + c * ld] = sh_beta;
    }
    __syncthreads();
  }
  if (blk == 0 && tid >= NT - B) t_column(ncol - 1);
  __syncthreads();
  if (blk == 0)  // (columns beyond the last reflector: zero)
    for (int t = tid; t < B * B; t += NT) {
      if (t / B >= ncol) a.Tm[t] = zero_<T>();
      else if (a.t_smem) a.Tm[t] = Ts[t];
    }
  // ---- write back: R (upper part) into the panel with zeros below, Y explicitly
  for (int idx = tid; idx < rows * B; idx += NT) {
    const int r = idx % rows, j = idx / rows;
    const int pr = lo + r;
    const T val = base[r + j * ld];
    const T y = (pr == j) ? from_re<T>(1.0) : (pr > j ? sc[j] * val : zero_<T>());
    const long long o = pr + j * a.ldy;
    a.Y[o] = y;
    a.Y1[o] = y;
    a.Y2[o] = y;
    a.Y3[o] = y;
    a.P[pr + j * a.ldp] = (pr <= j) ? val : zero_<T>();
  }
}

template <class T, int B, int CL> size_t panel_smem(int R, int use_smem, int t_smem) {
  constexpr int NT = panel_nt<B>();
  size_t s = (size_t)(NT + 3 * B) * sizeof(T) + (NT / 32 + NT / B) * sizeof(double) + 64;
  if (t_smem) s += (size_t)B * B * sizeof(T);
  if (CL) s += (size_t)(2 * CL * B + 2 * B) * sizeof(T) + 2 * CL * sizeof(double);
  if (use_smem) s += (size_t)(R | 1) * B * sizeof(T);
  return s;
}

constexpr int PANEL_CL = 16;  // blocks of the one-cluster form (beyond the portable 8: asked for and checked)

// Whether a panel of m rows goes to one cluster: its 16 SMs' FP64 pipe time for a column grows with m, the grid's
// barrier does not.  full->band of the two forms (ms, grid / best limit): real n = 256, b = 32 1.38 / 1.02, 1500
// 11.3 / 10.2 (limit 1000 to 2000), 3000 28.0 / 26.9 (1000 - 1500; 28.8 for all panels); b = 16 n = 2000 21.4 / 18.9 (from
// 2000); b = 64 n = 3000 29.4 / 26.2 (2000); complex b = 16 n = 2000 40.1 / 39.5 (1000), b = 32 31.1 / 30.7 (500); FP32
// n = 3000 22.9 / 22.2 (1000).
template <class T, int B> bool panel_in_cluster(int m) {
  const int lim = B == 16 ? 2400 : (B == 32 ? 1400 : 2000);
  return m < (is_cx<T>::value ? lim / 3 : lim);
}

// The QR of one panel (a.m rows): rows per block, residence in shared memory when it fits.
template <class T, int B> int launch_panel(Sys& s, PanelArgs<T> a, int* arrivals) {
  constexpr int NT = panel_nt<B>();
  const size_t cap = (size_t)200 * 1024;
  if (panel_in_cluster<T, B>(a.m)) {
    const auto kern = k_panel_qr<T, B, PANEL_CL>;
    a.R = (a.m + PANEL_CL - 1) / PANEL_CL;
    a.t_smem = a.use_smem = 1;
    const size_t smem = panel_smem<T, B, PANEL_CL>(a.R, 1, 1);
    if (smem <= cap) {
      GEV_TRY(allow_max_dyn_smem(kern));
      GEV_TRY(allow_wide_cluster(kern));
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = PANEL_CL;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(PANEL_CL);
      cfg.blockDim = dim3(NT);
      cfg.dynamicSmemBytes = smem;
      cfg.stream = s.stream;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int fit = 0;
      if (cudaOccupancyMaxActiveClusters(&fit, kern, &cfg) == cudaSuccess && fit >= 1) {
        GEV_COUNT(s);
        GEV_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, a));
        return 0;
      }
      cudaGetLastError();  // no cluster of this size here: the grid form
    }
  }
  GEV_TRY(allow_max_dyn_smem(k_panel_qr<T, B, 0>));
  // Blocks: a column costs a block 2 R / 4 b / 32 multiply-adds of FP64 pipe time for its R = m / G rows (twice
  // that for complex data against additions) and G / 4 b / 32 sums of a third of that time for the G partial sums: least
  // at G^2 = 6 m (12 m).
  int G = std::min(s.sms, (int)std::ceil(std::sqrt((is_cx<T>::value ? 12.0 : 6.0) * a.m))), per_sm = 0;
  a.R = std::max(8, (a.m + G - 1) / G);
  G = (a.m + a.R - 1) / a.R;
  a.t_smem = panel_smem<T, B, 0>(a.R, 0, 1) <= cap ? 1 : 0;
  a.use_smem = panel_smem<T, B, 0>(a.R, 1, a.t_smem) <= cap ? 1 : 0;
  if (!a.use_smem && panel_smem<T, B, 0>(a.R, 1, 0) <= cap) {
    a.t_smem = 0;
    a.use_smem = 1;
  }
  const size_t smem = panel_smem<T, B, 0>(a.R, a.use_smem, a.t_smem);
  GEV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_panel_qr<T, B, 0>, NT, smem));
  if (per_sm < 1 || G > per_sm * s.sms || G > 4096) return GEV_ERR_UNSUPPORTED;
  a.base = *arrivals;
  *arrivals += G * std::min(a.m, B);
  void* args[] = {&a};
  GEV_COUNT(s);
  GEV_CUDA_TRY(cudaLaunchCooperativeKernel((void*)k_panel_qr<T, B, 0>, dim3(G), dim3(NT), args, smem, s.stream));
  return 0;
}

// M (2b x b) = [T; -U / 2], U = T^H (Z T) for Z = Y^H W0 (b x b): one column per block of 4 b threads (four to
// an output, each a quarter of the sum), T in shared memory.  (As two products of b x b x b on the tensor-core
// engine: four launches.  Four columns per block took 17 us for b = 32 and 29 us for b = 64, one 5.9 and 9.3 us.)
template <class T>
__global__ void __launch_bounds__(256) k_sbr_coef(int b, const T* Z, const T* Tm, T* M) {
  extern __shared__ __align__(16) unsigned char smraw[];
  T* Ts = reinterpret_cast<T*>(smraw);  // b x b, ld b + 1
  T* red = Ts + b * (b + 1);            // 4 x b
  T* Q = red + 4 * b;                   // Z T(:, j)
  const int tid = threadIdx.x, j = blockIdx.x, i = tid % b, h = tid / b, kq = b / 4;
  for (int t = tid; t < b * b; t += 4 * b) Ts[t % b + (t / b) * (b + 1)] = Tm[t];
  __syncthreads();
  T acc = zero_<T>();
#pragma unroll 4
  for (int k = h * kq; k < (h + 1) * kq; ++k) mac(acc, Z[i + k * b], Ts[k + j * (b + 1)]);
  red[tid] = acc;
  __syncthreads();
  if (h == 0) Q[i] = (red[i] + red[b + i]) + (red[2 * b + i] + red[3 * b + i]);
  __syncthreads();
  acc = zero_<T>();
#pragma unroll 4
  for (int k = h * kq; k < (h + 1) * kq; ++k) cmac(acc, Ts[k + i * (b + 1)], Q[k]);
  red[tid] = acc;
  __syncthreads();
  if (h == 0) {
    M[i + j * 2 * b] = Ts[i + j * (b + 1)];
    M[b + i + j * 2 * b] = from_re<T>(-0.5) * ((red[i] + red[b + i]) + (red[2 * b + i] + red[3 * b + i]));
  }
}

// band[(i-j) + j*ldb] = A(i,j) for 0 <= i-j <= b, zero for b < i-j < ldb.
template <class T>
__global__ void k_extract_band(int n, int b, const T* A, long long lda, T* band, int ldb) {
  const long long total = (long long)n * ldb;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int d = (int)(t % ldb), j = (int)(t / ldb);
    const int i = j + d;
    T v = zero_<T>();
    if (d <= b && i < n) v = A[i + j * lda];
    if (d == 0) v = from_re<T>(re_(v));
    band[t] = v;
  }
}

}  // namespace

template <class T> int he2hb(Sys& s, T* A, int lda, int b) {
  const int n = s.n;
  T* V1 = (T*)s.V1;
  // the panels' reflector columns are stored from their own first row on; the rows above are zero so
  // that consecutive panels form one wider compact-WY block in the back-transform
  GEV_CUDA_TRY(cudaMemsetAsync(V1, 0, sizeof(T) * (size_t)n * n, s.stream));
  T* T1 = (T*)s.T1;
  const size_t buf = (size_t)n * 2 * b;      // the panel buffers, n x 2b each
  T* WY = (T*)s.Pn;                           // [W0 | Y]
  T* YV = WY + buf;                           // [Y | V]
  T* VY = YV + buf;                           // [V | Y]
  T* M = VY + buf;                            // 2b x b
  T* Z = (T*)s.small;
  double* nrm_part = (double*)s.panelws;     // 2 x 4096 (by column parity)
  T* prow = (T*)(nrm_part + 2 * 4096);        // 2 x b pivot rows
  T* w_part = prow + 2 * 128;                 // 2 x 4096 x b
  const T one = from_re<T>(1.0), mone = from_re<T>(-1.0), zero = zero_<T>();
  const size_t coef_smem = sizeof(T) * ((size_t)b * (b + 1) + 5 * b);
  GEV_TRY(allow_dyn_smem(k_sbr_coef<T>, coef_smem));
  // tasks of a sweep of the chase that follows.  V2 holds b n ntask entries for every b the handle accepts; the
  // scalars of a band narrower than its default outgrow their own room and go to Zk, which only complete solves (at the default width) use
  s.ntask = (n + b - 1) / b + 2;
  s.tau2 = s.ntask <= s.ntask_ws ? s.tau2_ws : (void*)s.Zk;
  if (s.ntask > s.ntask_ws && sizeof(T) * (size_t)s.ntask > sizeof(double) * (size_t)n) return GEV_ERR_UNSUPPORTED;
  int npanel = 0, arrivals = 0;
  GEV_CUDA_TRY(cudaMemsetAsync(&s.status[ST_BARRIER_CNT], 0, 2 * sizeof(int), s.stream));
  for (int j0 = 0;; j0 += b) {
    const int r0 = j0 + b;
    const int m = n - r0;
    if (m < 2) break;
    ++npanel;
    T* Yp = V1 + r0 + (long long)j0 * n;
    T* Tp = T1 + (long long)j0 * b;
    T* Wv = YV + (size_t)n * b;
    PanelArgs<T> a{};
    a.m = m;
    a.P = A + r0 + (long long)j0 * lda;
    a.ldp = lda;
    a.Y = Yp;
    a.Y1 = WY + (size_t)n * b;
    a.Y2 = YV;
    a.Y3 = VY + (size_t)n * b;
    a.ldy = n;
    a.Tm = Tp;
    a.nrm_part = nrm_part;
    a.w_part = w_part;
    a.prow = prow;
    a.count = &s.status[ST_BARRIER_CNT];
    a.status = s.status;
    a.abort_flag = &s.status[ST_ABORT];
    if (b == 16) GEV_TRY((launch_panel<T, 16>(s, a, &arrivals)));
    else if (b == 32) GEV_TRY((launch_panel<T, 32>(s, a, &arrivals)));
    else if (b == 64) GEV_TRY((launch_panel<T, 64>(s, a, &arrivals)));
    else return GEV_ERR_UNSUPPORTED;
    // ---- two-sided update of the trailing block: with W = A22 Y T, Z = Y^H A22 Y, U = T^H Z T,
    //      V = W - Y U / 2 = [A22 Y, Y] [T; -U / 2], the rank-2b update as ONE product:
    //      A22 -= Y V^H + V Y^H = [Y V] [V Y]^H  (K = 2b: the trailing block is read and written once)
    T* A22 = A + r0 + (long long)r0 * lda;
    gemm(s, gp<T>(m, b, m, 0, 0, one, A22, lda, Yp, n, zero, WY, n));  // W0 = A22 Y
    gemm(s, gp<T>(b, b, m, 2, 0, one, Yp, n, WY, n, zero, Z, b));      // Z = Y^H W0
    GEV_COUNT(s);
    k_sbr_coef<T><<<b, 4 * b, coef_smem, s.stream>>>(b, Z, Tp, M);
    GemmP<T> g = gp<T>(m, b, 2 * b, 0, 0, one, WY, n, M, 2 * b, zero, Wv, n);
    if (gemm_on_fp64_pipe(s, g)) {
      gemm(s, g);
    } else {  // (one product of both would scale W0 and Y, and T and U, together)
      g = gp<T>(m, b, b, 0, 0, one, WY, n, M, 2 * b, zero, Wv, n);
      g.tri_b = 2;
      gemm(s, g);
      gemm(s, gp<T>(m, b, b, 0, 0, one, Yp, n, M + b, 2 * b, one, Wv, n));
    }
    GEV_TRY(copy2d<T>(s, m, b, Wv, n, VY, n));
    g = gp<T>(m, m, 2 * b, 0, 2, mone, YV, n, VY, n, one, A22, lda);    // A22 -= [Y V] [V Y]^H
    g.c_lower = 1;
    gemm(s, g);
    GEV_TRY(mirror_lower<T>(s, m, A22, lda));
  }
  // ---- compact band for the bulge chasing
  const int ldb = 2 * b;
  if (ldb > s.ldband) return GEV_ERR_UNSUPPORTED;
  {
    long long total = (long long)n * ldb;
    unsigned blocks = cdiv(total, 256);
    if (blocks > 16u * s.sms) blocks = 16u * s.sms;
    GEV_COUNT(s);
    k_extract_band<T><<<blocks, 256, 0, s.stream>>>(n, b, A, lda, (T*)s.band, ldb);
    GEV_TRY(last_error());
  }
  s.band_b_used = b;
  s.have_band = true;
  s.have_tridiag_refl = false;
  s.nsbr_panels = npanel;
  s.q1_pw = b;
  s.q1_off = b;
  s.q1_nrefl = npanel * b;
  s.one_stage_used = false;
  return 0;
}

// Y <- Q1 Y (n x k), Q1 = Q_0 Q_1 ... Q_last: the panels' compact-WY blocks, applied G panels at a
// time.  Panel p holds reflectors p*pw .. p*pw + w_p - 1 (w_p = pw but for a narrower last panel of
// the one-stage reduction), stored in those columns of V1 from row p*pw + off on (off = b for the
// full -> band panels, 1 for the one-stage ones), each zero above its own first row (V1 is cleared
// before the reduction), with its w_p x w_p factor T_p at T1 + p pw^2 (ld pw).  Consecutive panels
// p .. p+G-1 merge into one block  Q_p ... Q_{p+G-1} = I - Yg Tg Yg^H,  Yg = [Y_p ... Y_{p+G-1}],
// Tg upper triangular, built block column by block column from the T_j and the Gram blocks Yg^H Yg:
//     Tg(0:o_j, o_j:o_j+w_j) = -Tg(0:o_j, 0:o_j) (Yg(:, 0:o_j)^H Y_j) T_j,   Tg(o_j.., o_j..) = T_j.
// Each group then costs three products with inner dimension sum w_j (or m), last group first.
template <class T> int bt_he2hb(Sys& s, T* Yb, int ldy, int k) {
  const int n = s.n, pw = s.q1_pw, off = s.q1_off, nrefl = s.q1_nrefl;
  T* V1 = (T*)s.V1;
  T* T1 = (T*)s.T1;
  const int np = s.nsbr_panels;
  if (np <= 0) return 0;
  const int G = std::min(4, np);
  const int gb = G * pw;                  // <= 4 b
  T* Wk = (T*)s.Pn;                       // gb x k  (the panel buffers: 8 b n elements)
  T* Wk2 = Wk + (size_t)gb * k;           // gb x k
  T* Tg = (T*)s.btg;                      // gb x gb
  T* Gg = Tg + (size_t)gb * gb;           // gb x gb Gram blocks
  T* Xg = Gg + (size_t)gb * gb;           // gb x pw
  const T one = from_re<T>(1.0), mone = from_re<T>(-1.0), zero = zero_<T>();
  auto width = [&](int p) { return std::min(pw, nrefl - p * pw); };
  const int ngroups = (np + G - 1) / G;
  for (int q = ngroups - 1; q >= 0; --q) {
    const int p0 = q * G, pc = std::min(G, np - p0);
    int w = 0;
    for (int j = 0; j < pc; ++j) w += width(p0 + j);
    const int j0 = p0 * pw, r0 = j0 + off, m = n - r0;
    if (m <= 0 || w <= 0) continue;
    const T* Yg = V1 + r0 + (long long)j0 * n;  // m x w
    // Tg: block column 0 = T_p0; block column j from the Gram blocks
    GEV_CUDA_TRY(cudaMemset2DAsync(Tg, sizeof(T) * gb, 0, sizeof(T) * w, w, s.stream));
    GEV_TRY(copy2d<T>(s, width(p0), width(p0), T1 + (size_t)p0 * pw * pw, pw, Tg, gb));
    if (pc > 1) {
      GemmP<T> g = gp<T>(w, w, m, 2, 0, one, Yg, n, Yg, n, zero, Gg, gb);  // Gram Yg^H Yg
      gemm(s, g);
      for (int j = 1; j < pc; ++j) {
        const int oj = j * pw, wj = width(p0 + j);
        const T* Tj = T1 + (size_t)(p0 + j) * pw * pw;
        g = gp<T>(oj, wj, wj, 0, 0, one, Gg + (size_t)oj * gb, gb, Tj, pw, zero, Xg, gb);  // X = G(0:oj, j) T_j
        g.tri_b = 2;
        gemm(s, g);
        g = gp<T>(oj, wj, oj, 0, 0, mone, Tg, gb, Xg, gb, zero, Tg + (size_t)oj * gb, gb);
        g.tri_a = 2;                                                   // Tg(0:oj, j) = -Tg(0:oj, 0:oj) X
        gemm(s, g);
        GEV_TRY(copy2d<T>(s, wj, wj, Tj, pw, Tg + oj + (size_t)oj * gb, gb));
      }
    }
    T* Ysub = Yb + r0;
    gemm(s, gp<T>(w, k, m, 2, 0, one, Yg, n, Ysub, ldy, zero, Wk, gb));  // Wk = Yg^H Y
    GemmP<T> g = gp<T>(w, k, w, 0, 0, one, Tg, gb, Wk, gb, zero, Wk2, gb);  // Wk2 = Tg Wk
    g.tri_a = 2;
    gemm(s, g);
    gemm(s, gp<T>(m, k, w, 0, 0, mone, Yg, n, Wk2, gb, one, Ysub, ldy));  // Y -= Yg Wk2
  }
  return last_error();
}

// Step 6 ("Back"): Y = Q1 Q2 D Z.
template <class T> int back(Sys& s, const double* Z, int ldz, int k, T* Y, int ldy) {
  if (s.one_stage_used) return back_td<T>(s, Z, ldz, k, Y, ldy);
  GEV_TRY(bt_hb2st<T>(s, Z, ldz, k, Y, ldy));
  GEV_TRY(bt_he2hb<T>(s, Y, ldy, k));
  return 0;
}

template int back<double>(Sys&, const double*, int, int, double*, int);
template int back<zd>(Sys&, const double*, int, int, zd*, int);
template int he2hb<double>(Sys&, double*, int, int);
template int he2hb<zd>(Sys&, zd*, int, int);
template int bt_he2hb<double>(Sys&, double*, int, int);
template int he2hb<float>(Sys&, float*, int, int);
template int bt_he2hb<float>(Sys&, float*, int, int);
template int bt_he2hb<zd>(Sys&, zd*, int, int);

}  // namespace gev
