// Stage 2 of the two-stage tridiagonalisation: band (width b) -> real symmetric tridiagonal by
// bulge chasing, B = Q2 T' Q2^H, and the back-transform Y = Q2 D Z (D: diagonal phases that make
// the complex off-diagonal real).
//
// Sweep s (s = 0 .. n-3) annihilates column s below the subdiagonal with a Householder reflector
// H(s,0) on rows W_0 = [s+1, s+1+b); applying it two-sided fills the b x b block below the window
// (the bulge).  Task t >= 1 annihilates the first column of that block with H(s,t) on rows
// W_t = [s+1+tb, s+1+(t+1)b), and so on down the band.  Footprint of task (s,t): rows
// [p_t, p_{t+2}), columns [p_{t-1}, p_{t+1}) (p_t = s+1+tb).  Task (s+1,t) overlaps tasks
// (s,t-1) .. (s,t+2) only, and of (s,t+2) only the entry (p_{t+2}, p_{t+1}) that its reflector fixes, so
// sweep s+1 may run task t once sweep s has finished task t+1 and formed the reflector of task t+2.
//
// GPU mapping: one persistent cooperative kernel; block q owns sweeps q, q+G, q+2G, ... and runs
// their tasks in order, staging the three blocks of a task (L = (W_t, W_{t-1}), D = (W_t, W_t),
// E = (W_{t+1}, W_t)) in shared memory; E stays resident as the next task's L.  A per-sweep
// progress counter (release store, acquire load, band reads through L2 with __ldcg) orders the sweeps.  Every wait is bounded (status[ST_SPIN] iterations
// when the host set a limit, else kSpinLimit, ~2 s): on expiry the kernel records ST_TIMEOUT, raises
// the abort flag and all blocks return.
//
// The band is stored compactly: element (i, j), 0 <= i-j < 2b, at band[(i-j) + j*ldb], ldb = 2b
// (rows b+1 .. 2b-1 below the diagonal hold the bulge).
#include <algorithm>
#include <climits>

#include <type_traits>

#include "common.cuh"
#include "coop.cuh"

namespace gev {

namespace {

__device__ __forceinline__ double warp_sum(double v) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}
__device__ __forceinline__ zd warp_sum(zd v) { return make_zd(warp_sum(v.x), warp_sum(v.y)); }
__device__ __forceinline__ float warp_sum(float v) {
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  return v;
}
__device__ __forceinline__ zf warp_sum(zf v) { return make_zf(warp_sum(v.x), warp_sum(v.y)); }

// Bounded acquire-wait of one warp until *flag >= target; false on timeout / abort.
__device__ __forceinline__ bool warp_wait_ge(const int* flag, int target, int* status, int* abort_flag, int site) {
  int good = 1;
  if ((threadIdx.x & 31) == 0 && ld_acquire(flag) < target) {
    volatile int* va = abort_flag;
    const long long lim = spin_limit(status);
    long long it = 0;
    while (ld_acquire(flag) < target) {
      if (*va) { good = 0; break; }
      if (++it > lim) {
        atomicCAS(&status[ST_TIMEOUT], 0, site);
        atomicExch(abort_flag, 1);
        good = 0;
        break;
      }
      if (it > 16) __nanosleep(32);
    }
  }
  return __shfl_sync(0xffffffffu, good, 0) != 0;
}

__device__ __forceinline__ void bar_sync_n(int id, int n) { asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }
__device__ __forceinline__ void bar_arrive_n(int id, int n) { asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(n) : "memory"); }

// Band -> tridiagonal by bulge chasing (one sweep per block at a time).  Task t of sweep s
// annihilates the column below the band with one Householder reflector H = I - tau v v^H
// (v_0 = 1) acting on rows p .. p+len-1, p = s + 1 + t b:
//   L (the block left of the reflector's rows, the previous task's bulge) <- H L   (t > 0),
//   D (the diagonal block)                                                  <- H D H^H,
//   E (the block below D: the new bulge)                                    <- E H^H,
// and the reflector is kept for back-transform 2.
//
// The chase is one chain of dependent steps per sweep, and the sweeps follow one another at a fixed
// lag, so the run time is (lag in tasks) x (time of a task) x n.  Both are kept short:
//  * Lag.  Task (s+1, t) reads what the tasks (s, 0 .. t+1) leave, and of task (s, t+2) only the one
//    entry of the band that its reflector makes (beta, at row p_{t+2}, column p_{t+1}).  Progress t+3
//    is therefore published when the REFLECTOR of task t+2 is known, not when the task is done: the
//    lag is two tasks and a reflector instead of three tasks.
//  * Task.  The products w = v^H L, y = D v, z = E v depend on v only, so they run as one phase (all
//    warps equally: on GB300 the FP64 pipe, about 1.6 FMA per SM per cycle, bounds this kernel), their
//    sums as a second, the three updates as a third.  Column 0 of the updated E, the next
//    reflector's x, is E(:,0) - z (v_0 = 1): it comes out of the second phase, so warp 0 computes the
//    next reflector (reduction, rsqrt, reciprocal: a long latency chain) while the other warps
//    update, wait for the next task's blocks and load them.  A warp of its own publishes the progress as
//    soon as the stores of this task are done (a barrier that the others only arrive at): the release waits
//    about 1000 cycles for the stores, in the middle of the chain when warp 0 issued it.
//    Warp 1 finishes y (its inner product with v) while the rest update L and E.
//  * Four barriers per task; D and E travel through registers, so that no wait holds the others up.
// Measured (to_tridiag; one barrier-separated product after another, a lag of three tasks and the release in
// warp 0 at first): real FP64 n = 10240, b = 64 447 -> 190 ms (bound by the FP64 pipe: 14000 of a task's 16000
// cycles), n = 1500, b = 32 37.1 -> 12.2 ms; complex FP64 n = 509 29.7 -> 9.4 ms; FP32 n = 6144 82.9 -> 40 ms.
// All arithmetic is in the data's own precision (FP32 for the mixed form).
template <class T, int B, int NTH>
__global__ void __launch_bounds__(NTH + 32) k_bulge(int n, T* band, int ldb, T* V2, T* tau2, int ntask, int* progress,
                                               int* status, int* abort_flag, int stall) {
  using R = typename real_of<T>::type;
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int LD = B + 1, O3 = 3 * B, P = NTH / O3, TERMS = B / P, NL = NTH - 32;
  constexpr int PF = (B * B + NL - 1) / NL;  // register slots per loading thread (D and E each)
  static_assert(NTH % 32 == 0 && NTH == P * O3 && B % P == 0 && (B * B) % 32 == 0, "thread mapping");
  T* Ls = reinterpret_cast<T*>(smraw);
  T* Es = Ls + B * LD;
  T* Ds = Es + B * LD;
  T* vbuf = Ds + B * LD;      // 2 x B: the reflector of this and of the next task
  T* vc = vbuf + 2 * B;       // conj(v)
  T* w = vc + B;              // L: conj(tau) v^H L
  T* y = w + B;               // D: tau D v - c v
  T* z = y + B;               // E: tau E v
  T* xn_ = z + B;             // column 0 of the updated E: the next task's x
  T* part = xn_ + B;          // P x 3B partial sums
  __shared__ T sh_tau[2];
  __shared__ volatile int bad;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) bad = 0;
  __syncthreads();

  // The publisher (the last warp): waits for the stores of a task (barrier 1, where the others only arrive) and
  // releases the sweep's progress.  Barrier 3, in the middle of a task, keeps the others from completing barrier 1
  // twice before it has left it once.
  if (warp == NTH / 32) {
    for (int s = blockIdx.x; s <= n - 3; s += gridDim.x)
      for (int t = 0;; ++t) {
        const int pn = s + 1 + t * B + B;
        const bool more = pn < n && min(B, n - pn) > 1;
        bar_sync_n(3, NTH + 32);
        if (bad) return;
        bar_sync_n(1, NTH + 32);
        if (bad) return;
        if (lane == 0) st_release(&progress[s], more ? t + 2 : INT_MAX);
        if (!more) break;
      }
    return;
  }

  // warp 0: the reflector of the B entries x (zero beyond len) -> v, conj(v) is formed with the loads
  auto reflect = [&](const T* x, T* v, int slot) {
    T xv[(B + 31) / 32];
    R s2 = 0;
#pragma unroll
    for (int u = 0; u < (B + 31) / 32; ++u) {
      const int i = lane + 32 * u;
      xv[u] = i < B ? x[i] : zero_<T>();
      if (i > 0) s2 += (R)abs2_(xv[u]);
    }
    s2 = warp_sum(s2);
    const T alpha = x[0];
    T tau = zero_<T>(), beta = alpha, scale = zero_<T>();
    if (!(is_zero(s2) && im_(alpha) == 0)) house(alpha, s2, tau, beta, scale);
#pragma unroll
    for (int u = 0; u < (B + 31) / 32; ++u) {
      const int i = lane + 32 * u;
      if (i < B) v[i] = i == 0 ? from_re<T>(1.0) : scale * xv[u];
    }
    if (lane == 0) sh_tau[slot] = tau;
    return beta;
  };

  for (int s = blockIdx.x; s <= n - 3; s += gridDim.x) {
    T dreg[PF], ereg[PF];
    // wait for the blocks of task t and load D (lower triangle) and E into registers (warps 1 ..)
    auto fetch = [&](int t) {
      const int p = s + 1 + t * B, len = min(B, n - p), p2 = p + len, len2 = min(B, n - p2);
      bool ok = true;
      if (s > 0)
        ok = stall ? warp_wait_ge(&status[ST_STALL], 1, status, abort_flag, 202)
                   : warp_wait_ge(&progress[s - 1], t + 3, status, abort_flag, 201);
      if (!ok) {
        if (lane == 0) bad = 1;
        return;
      }
#pragma unroll
      for (int u = 0; u < PF; ++u) {
        const int idx = tid - 32 + u * NL, i = idx & (B - 1), j = idx / B;
        const T* col = band + (long long)(p + j) * ldb;
        dreg[u] = (idx < B * B && j < len && i < len && i >= j) ? ldcg_(&col[i - j]) : zero_<T>();
        ereg[u] = (idx < B * B && j < len && i < len2) ? ldcg_(&col[len + i - j]) : zero_<T>();
      }
    };
    int cur = 0;
    // ---- the sweep's first reflector: column s below the diagonal
    if (warp == 0) {
      bool ok = true;
      if (s > 0)
        ok = stall ? warp_wait_ge(&status[ST_STALL], 1, status, abort_flag, 202)
                   : warp_wait_ge(&progress[s - 1], 3, status, abort_flag, 201);
      if (!ok) {
        if (lane == 0) bad = 1;
      } else {
        const int len = min(B, n - s - 1);
        T* col = band + (long long)s * ldb + 1;
        for (int i = lane; i < B; i += 32) xn_[i] = i < len ? ldcg_(&col[i]) : zero_<T>();
        __syncwarp();
        const T beta = reflect(xn_, vbuf, 0);
        for (int i = lane; i < len; i += 32) stcg_(&col[i], i == 0 ? beta : zero_<T>());
      }
    } else {
      fetch(0);
    }
    for (int t = 0;; ++t) {
      const int p = s + 1 + t * B, len = min(B, n - p), p2 = p + len, len2 = min(B, n - p2);
      const int pn = p + B, lenn = pn < n ? min(B, n - pn) : 0;  // the next task's rows
      const bool more = lenn > 1;
      T* v = vbuf + cur * B;
      T* vn = vbuf + (cur ^ 1) * B;
      // ---- D and E to shared memory
      if (warp > 0) {
#pragma unroll
        for (int u = 0; u < PF; ++u) {
          const int idx = tid - 32 + u * NL, i = idx & (B - 1), j = idx / B;
          if (idx < B * B) {
            if (i >= j) {
              const T val = i == j ? from_re<T>(re_(dreg[u])) : dreg[u];
              Ds[i + j * LD] = val;
              Ds[j + i * LD] = conj_(val);
            }
            Es[i + j * LD] = ereg[u];
          }
        }
      } else {
        __syncwarp();
        for (int i = lane; i < B; i += 32) vc[i] = conj_(v[i]);
      }
      bar_sync_n(0, NTH);
      if (bad) {  // (uniform: set before the barrier, never cleared)
        bar_arrive_n(3, NTH + 32);
        return;
      }
      const T tau = sh_tau[cur];
      // ---- partial sums of w = v^H L, y = D v, z = E v: P threads per output
      {
        const int o = tid % O3, g = tid / O3, i = o & (B - 1), m = o / B;
        const T* a = m == 0 ? Ls + i * LD : (m == 1 ? Ds + i : Es + i);
        const T* x = m == 0 ? vc : v;
        const int st = m == 0 ? 1 : LD, j0 = g * TERMS;
        T acc = zero_<T>(), acc2 = zero_<T>();
        if (m == 1 || (m == 0 ? t > 0 : len2 > 0)) {
#pragma unroll 8
          for (int j = 0; j < TERMS; j += 2) {
            mac(acc, a[(j0 + j) * st], x[j0 + j]);
            mac(acc2, a[(j0 + j + 1) * st], x[j0 + j + 1]);
          }
        }
        part[tid] = acc + acc2;
      }
      bar_sync_n(0, NTH);
      for (int o = tid; o < O3; o += NTH) {
        T acc = part[o];
#pragma unroll
        for (int g = 1; g < P; ++g) acc += part[g * O3 + o];
        const int i = o & (B - 1), m = o / B;
        if (m == 0) w[i] = conj_(tau) * acc;
        else if (m == 1) y[i] = acc;
        else {
          const T zz = tau * acc;
          z[i] = zz;
          xn_[i] = Es[i] - zz;
        }
      }
      bar_sync_n(3, NTH + 32);
      if (warp == 0) {
        // ---- the next reflector, published once this task's stores are done
        if (more) {
          const T beta = reflect(xn_, vn, cur ^ 1);
          if (lane == 0) stcg_(&band[B + (long long)p * ldb], beta);
        }
        __syncwarp();
        if (more) bar_arrive_n(1, NTH + 32);
      } else {
        if (warp == 1) {
          // y <- tau y - c v, c = |tau|^2 Re(v^H y) / 2
          T yv[(B + 31) / 32], vv[(B + 31) / 32];
          R acc = 0;
#pragma unroll
          for (int u = 0; u < (B + 31) / 32; ++u) {
            const int i = lane + 32 * u;
            yv[u] = i < B ? y[i] : zero_<T>();
            vv[u] = i < B ? v[i] : zero_<T>();
            acc += (R)re_(cmul(vv[u], yv[u]));
          }
          acc = warp_sum(acc);
          const T c = from_re<T>((R)0.5 * (R)abs2_(tau) * acc);
#pragma unroll
          for (int u = 0; u < (B + 31) / 32; ++u) {
            const int i = lane + 32 * u;
            if (i < B) y[i] = tau * yv[u] - c * vv[u];
          }
        } else {
          // L <- H L, stored (its column 0 is beta, 0 ..; beta was stored with the reflector); E <- E H^H
          // (column 0 is xn_, consumed by the next reflector); the reflector for the back-transform
          constexpr int NW = NTH - 64;
          for (int idx = tid - 64; idx < B * B; idx += NW) {
            const int i = idx & (B - 1), q = idx / B;
            if (t > 0 && i < len && (q > 0 || i > 0)) {
              T val = zero_<T>();
              if (q > 0) {
                val = Ls[i + q * LD];
                nmac(val, v[i], w[q]);
              }
              stcg_(&band[(B + i - q) + (long long)(p - B + q) * ldb], val);
            }
            if (q > 0 && len2 > 0) nmacc(Es[i + q * LD], z[i], v[q]);
          }
          const long long rid = (long long)s * ntask + t;
          for (int i = tid - 64; i < B; i += NW) V2[rid * B + i] = v[i];
          if (tid == 64) tau2[rid] = tau;
        }
        bar_sync_n(2, NL);
        // D <- H D H^H, lower triangle: columns c and B - 1 - c together have B - 1 entries below the
        // diagonal, so a pair fills whole warps; then the diagonal
        for (int idx = tid - 32; idx < (B / 2) * B; idx += NL) {
          const int c = idx / B, e = idx & (B - 1);
          const bool first = e < B - 1 - c;
          const int i = first ? c + 1 + e : e + 1, j = first ? c : B - 1 - c;
          if (e < B - 1 && i < len && j < len) {
            T val = Ds[i + j * LD];
            nmacc(val, y[i], v[j]);
            nmacc(val, v[i], y[j]);
            stcg_(&band[(i - j) + (long long)(p + j) * ldb], val);
          }
        }
        for (int i = tid - 32; i < len; i += NL)
          stcg_(&band[(long long)(p + i) * ldb],
                from_re<T>(re_(Ds[i + i * LD]) - (R)2 * (R)re_(mulc(y[i], v[i]))));
        __syncwarp();
        if (more) {
          bar_arrive_n(1, NTH + 32);
          fetch(t + 1);
          bar_sync_n(2, NL);  // every warp has left D, E and L: the next task may overwrite them
        }
      }
      if (!more) {
        // a last single row below: store its part of the bulge
        if (lenn == 1) {
          if (warp > 0) {
            bool ok = true;
            if (s > 0)
              ok = stall ? warp_wait_ge(&status[ST_STALL], 1, status, abort_flag, 202)
                         : warp_wait_ge(&progress[s - 1], t + 4, status, abort_flag, 201);
            if (!ok && lane == 0) bad = 1;
            if (ok)
              for (int q = tid - 32; q < B; q += NL)
                stcg_(&band[(B - q) + (long long)(p + q) * ldb], q == 0 ? xn_[0] : Es[q * LD]);
          }
        }
        __syncwarp();
        bar_arrive_n(1, NTH + 32);
        break;
      }
      T* tmp = Ls;
      Ls = Es;
      Es = tmp;
      cur ^= 1;
    }
    bar_sync_n(0, NTH);
    if (bad) return;
  }
}

// d = Re diag, e = |subdiag| with the phase recursion phi_0 = 1, phi_{i+1} = phi_i eps_i/|eps_i|
// (complex), or e = subdiag (real).  One block of 1024 threads.  The phases are a running product:
// every thread forms the product of its own n / 1024 factors, the block scans the 1024 products in
// shared memory (10 steps), and the threads write their phases.  (As one thread's recursion the chain of
// n hypot's and divisions took about 2 us per row.)  The phases are formed in FP64 also from an FP32
// band, so that their product over n steps stays accurate.
template <class T>
__global__ void __launch_bounds__(1024) k_tridiag_out(int n, const T* band, int ldb, double* d, double* e, zd* phase) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) d[i] = re_(band[(long long)i * ldb]);
  if constexpr (is_cx<T>::value) {
    __shared__ zd sc[2][1024];
    const int tid = threadIdx.x, per = (n + 1023) / 1024, i0 = tid * per, i1 = min(n - 1, i0 + per);
    zd ph = make_zd(1.0, 0.0);
    for (int i = i0; i < i1; ++i) {  // the product of this thread's factors; phase[i + 1] = it, so far
      const T eps = band[1 + (long long)i * ldb];
      const double ex = re_(eps), ey = im_(eps);
      const double a = hypot(ex, ey);
      e[i] = a;
      if (a > 0.0) ph = ph * make_zd(ex / a, ey / a);
      phase[i + 1] = ph;
    }
    int cur = 0;
    sc[0][tid] = ph;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
      const zd v = sc[cur][tid];
      sc[cur ^ 1][tid] = tid >= off ? sc[cur][tid - off] * v : v;
      cur ^= 1;
      __syncthreads();
    }
    if (tid == 0) phase[0] = make_zd(1.0, 0.0);
    if (tid > 0) {
      const zd before = sc[cur][tid - 1];
      for (int i = i0; i < i1; ++i) phase[i + 1] = before * phase[i + 1];
    }
  } else {
    for (int i = threadIdx.x; i + 1 < n; i += blockDim.x) e[i] = band[1 + (long long)i * ldb];
  }
}

// Y = D Z (real Z -> scalar type; D = diag(phase) for complex data, identity for real).
template <class T>
__global__ void k_phase_rows(int n, int k, const double* Z, long long ldz, const zd* phase, T* Y,
                             long long ldy) {
  const long long total = (long long)n * k;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(t % n), c = (int)(t / n);
    const double z = Z[i + c * ldz];
    if constexpr (is_cx<T>::value) {
      const zd v = z * phase[i];
      Y[i + c * ldy] = T{(decltype(T{}.x))v.x, (decltype(T{}.x))v.y};
    } else {
      Y[i + c * ldy] = (T)z;
    }
  }
}

// Y <- Q2 Y, level-parallel.  With G = b sweeps per group, the block D_t^g of group g
// (reflectors H(s, t), s = gb .. gb+b-1, applied in the order s descending) acts on the row window
// [(g+t) b + 1, (g+t+2) b - 1).  Q2 = P_0 P_1 ... with P_g = D_T^g ... D_1^g D_0^g, so Y <- Q2 Y
// applies D_0^last first.  D_t^g must follow D_{t-1}^g and D_{t'}^{g+1} for t' <= t (overlapping
// windows), which is exactly the order of the levels L = t + (ngroups - 1 - g); blocks of one level
// have windows 2b apart, act on disjoint rows and commute.  One launch per level: blockIdx.x picks
// the group, blockIdx.y a share of Y's columns.
//
// A column is held by 8 lanes, lane r the window rows r, r + 8, ...; the reflectors are taken in chunks of
// 8 (descending), whose rows [8a, 8a + B + 7) are B / 8 + 1 registers per lane: after a chunk the
// topmost row of every lane is final and is stored, the others move up one register and the next row, loaded
// before the chunk, enters.  Nothing but the reflectors is staged in shared memory (shifted by q mod 8 and
// zero-padded, so that every chunk is the same straight-line code).  What bounds it is the FP64 pipe
// (1.25 b n k multiply-adds per level, four times that for complex data, at 4.5e11 per second over the
// chip) once there are enough columns, and the chain of b dot products (three shuffles each) before that.
// (One thread per column and 128 columns per block, as before, used nblk * ceil(k / 128) SMs.)  Back-transform 2,
// before -> now: complex n = 509, k = 128, b = 32 14.1 -> 2.8 ms; real n = 256, all pairs 2.2 -> 0.4 ms; complex64
// n = 1536, all vectors 7.5 -> 2.3 ms; real n = 1500, k = 375 9.0 (in tensor-core form) -> 4.5 ms.
constexpr int BTL_COLS = 16;
__device__ __forceinline__ float sum8(float v) {
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double sum8(double v) {
  for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ zd sum8(zd v) { return make_zd(sum8(v.x), sum8(v.y)); }
__device__ __forceinline__ zf sum8(zf v) { return make_zf(sum8(v.x), sum8(v.y)); }

template <class T, int B>
__global__ void __launch_bounds__(8 * BTL_COLS) k_bt_level(int n, int k, int L, int ngroups, const T* V2,
                                                           const T* tau2, int ntask, T* Y, long long ldy) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int LV = B + 8, NR = B / 8, NTH = 8 * BTL_COLS;
  T* Vs = reinterpret_cast<T*>(smraw);  // B x LV: entry q LV + x is v_q at window row 8 (q / 8) + x
  T* ts = Vs + B * LV;                  // B
  const int g = max(0, ngroups - 1 - L) + blockIdx.x;
  const int t = L - (ngroups - 1 - g);
  if (g >= ngroups || t < 0 || t >= ntask) return;
  const int s0 = g * B, w0 = s0 + 1 + t * B;
  if (w0 >= n) return;
  const int tid = threadIdx.x;
  for (int q = tid; q < B; q += NTH) ts[q] = s0 + q <= n - 3 ? tau2[(long long)(s0 + q) * ntask + t] : zero_<T>();
  __syncthreads();
  for (int idx = tid; idx < B * LV; idx += NTH) {
    const int q = idx / LV, rel = idx % LV - (q & 7);
    T v = zero_<T>();
    if (rel >= 0 && rel < B && w0 + q + rel < n && ts[q] != zero_<T>())
      v = V2[((long long)(s0 + q) * ntask + t) * B + rel];
    Vs[idx] = v;
  }
  __syncthreads();
  const int r = tid & 7, cl = tid >> 3;
  for (int cb = blockIdx.y * BTL_COLS; cb < k; cb += gridDim.y * BTL_COLS) {
    const bool cok = cb + cl < k;
    T* y = Y + w0 + r + (long long)(cb + cl) * ldy;
    const int left = cok ? n - w0 - r : 0;  // rows of this lane: offsets 8 j < left
    T z[NR + 1];
#pragma unroll
    for (int i = 0; i <= NR; ++i) {
      const int o = 8 * (NR - 1 + i);
      z[i] = o < left ? y[o] : zero_<T>();
    }
#pragma unroll 1
    for (int a = NR - 1; a >= 0; --a) {
      T nx = zero_<T>();
      if (a > 0 && 8 * (a - 1) < left) nx = y[8 * (a - 1)];
#pragma unroll
      for (int u = 7; u >= 0; --u) {
        const T* vq = Vs + (8 * a + u) * LV + r;
        T acc0 = zero_<T>(), acc1 = zero_<T>();
#pragma unroll
        for (int i = 0; i <= NR; ++i) {
          if (i & 1) cmac(acc1, vq[8 * i], z[i]);
          else cmac(acc0, vq[8 * i], z[i]);
        }
        const T w = ts[8 * a + u] * sum8(acc0 + acc1);
#pragma unroll
        for (int i = 0; i <= NR; ++i) nmac(z[i], vq[8 * i], w);
      }
      if (8 * (a + NR) < left) y[8 * (a + NR)] = z[NR];
      if (a > 0) {
#pragma unroll
        for (int i = NR; i > 0; --i) z[i] = z[i - 1];
        z[0] = nx;
      } else {
#pragma unroll
        for (int i = 0; i < NR; ++i)
          if (8 * i < left) y[8 * i] = z[i];
      }
    }
  }
}

// FP32 form of the level kernel: the same (group, task) blocks and level order, but each thread
// applies the reflectors to its column from registers.  The 64 reflectors of a block are taken in
// chunks of 8 (descending): a chunk touches window rows [q0, q0 + B + 7), which are moved from the
// staged shared-memory window into registers, updated by the 8 reflectors (dot products with four
// partial sums) and written back.  Reflector entries are shared-memory broadcasts, zero-padded
// beyond the matrix end, so every chunk runs the same straight-line code.
constexpr int BTF_COLS = 128, BTF_CH = 8;
template <int B>
__global__ void __launch_bounds__(BTF_COLS) k_bt_level_f32(int n, int k, int L, int ngroups, const float* V2,
                                                           const float* tau2, int ntask, float* Y, long long ldy) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int g = max(0, ngroups - 1 - L) + blockIdx.x;
  const int t = L - (ngroups - 1 - g);
  if (g >= ngroups || t < 0 || t >= ntask) return;
  const int s0 = g * B;
  const int s1 = min(s0 + B - 1, n - 3);
  const int w0 = s0 + 1 + t * B;
  if (w0 >= n) return;
  const int rows = min(n, s1 + 1 + t * B + B) - w0;  // <= 2B - 1
  constexpr int LDZ = BTF_COLS + 1;
  float* Zs = reinterpret_cast<float*>(smraw);          // 2B x LDZ
  float* Vs = Zs + 2 * B * LDZ;                          // B x B (16-byte aligned rows)
  float* ts = Vs + B * B;                                // B
  const int c0 = blockIdx.y * BTF_COLS;
  const int ncols = min(BTF_COLS, k - c0);
  for (int idx = threadIdx.x; idx < B * B; idx += BTF_COLS) {
    const int q = idx / B, i = idx % B;
    const int p = s0 + q + 1 + t * B;
    float v = 0.f;
    if (s0 + q <= s1 && i < n - p) v = V2[((long long)(s0 + q) * ntask + t) * B + i];
    Vs[idx] = v;
  }
  for (int q = threadIdx.x; q < B; q += BTF_COLS) ts[q] = (s0 + q <= s1) ? tau2[(long long)(s0 + q) * ntask + t] : 0.f;
  for (int idx = threadIdx.x; idx < 2 * B * BTF_COLS; idx += BTF_COLS) {
    const int r = idx % (2 * B), c = idx / (2 * B);  // consecutive threads: consecutive rows
    float v = 0.f;
    if (r < rows && c < ncols) v = Y[(w0 + r) + (long long)(c0 + c) * ldy];
    Zs[r * LDZ + c] = v;
  }
  __syncthreads();
  const int c = threadIdx.x;
  for (int q0 = B - BTF_CH; q0 >= 0; q0 -= BTF_CH) {
    float z[B + BTF_CH - 1];
#pragma unroll
    for (int j = 0; j < B + BTF_CH - 1; ++j) z[j] = Zs[(q0 + j) * LDZ + c];
#pragma unroll
    for (int u = BTF_CH - 1; u >= 0; --u) {
      const float4* v4 = reinterpret_cast<const float4*>(Vs + (q0 + u) * B);
      float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
      for (int i = 0; i < B / 4; ++i) {
        const float4 v = v4[i];
        a0 = fmaf(v.x, z[u + 4 * i], a0);
        a1 = fmaf(v.y, z[u + 4 * i + 1], a1);
        a2 = fmaf(v.z, z[u + 4 * i + 2], a2);
        a3 = fmaf(v.w, z[u + 4 * i + 3], a3);
      }
      const float w = ts[q0 + u] * ((a0 + a1) + (a2 + a3));
#pragma unroll
      for (int i = 0; i < B / 4; ++i) {
        const float4 v = v4[i];
        z[u + 4 * i] = fmaf(-v.x, w, z[u + 4 * i]);
        z[u + 4 * i + 1] = fmaf(-v.y, w, z[u + 4 * i + 1]);
        z[u + 4 * i + 2] = fmaf(-v.z, w, z[u + 4 * i + 2]);
        z[u + 4 * i + 3] = fmaf(-v.w, w, z[u + 4 * i + 3]);
      }
    }
#pragma unroll
    for (int j = 0; j < B + BTF_CH - 1; ++j) Zs[(q0 + j) * LDZ + c] = z[j];
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < 2 * B * BTF_COLS; idx += BTF_COLS) {
    const int r = idx % (2 * B), cc = idx / (2 * B);
    if (r < rows && cc < ncols) Y[(w0 + r) + (long long)(c0 + cc) * ldy] = Zs[r * LDZ + cc];
  }
}

// Compact-WY form of one level's reflector blocks, for the tensor-core back-transform: for block j
// (group g = g_lo + j, task t) with reflectors v_q = V(:, q) of sweeps s0 + q on the window rows
// [w0, w0 + 2b) (v_q non-zero in rows q .. q + b - 1, v_q(q) = 1),
//   D_j = H(s0) H(s0 + 1) ... H(s0 + b - 1) = I - V T V^H,  T upper triangular:
//   T_qq = tau_q,  T(0:q, q) = -tau_q T(0:q, 0:q) (V(:, 0:q)^H v_q),
// and W_j = V T (2b x b, column-major at W + j 2b b) is written for the second product.  A reflector
// with tau = 0 (a task that never ran) is a zero column.  One block of 256 threads per D_j: the Gram
// entries V^H V by all threads (padded shared-memory columns), the recurrence by one warp, W by all.
// The blocks of level L: groups g in [g_lo, g_lo + nblk) with task t = L - (ngroups - 1 - g) in
// range and a window start w0(g) = (2g + L - ngroups + 1) b + 1 below n; w00 = w0(g_lo); windows are
// 2b apart.  (Host and device.)
struct LevelBlocks {
  int g_lo, nblk, w00;
};
__host__ __device__ inline LevelBlocks level_blocks(int n, int b, int L, int ngroups, int ntask) {
  LevelBlocks lb{0, 0, 0};
  const int g_lo = max(0, ngroups - 1 - L);
  int g_hi = min(ngroups - 1, ntask - 1 + ngroups - 1 - L);
  while (g_hi >= g_lo && (2 * g_hi + L - ngroups + 1) * b + 1 >= n) --g_hi;
  if (g_hi < g_lo) return lb;
  lb.g_lo = g_lo;
  lb.nblk = g_hi - g_lo + 1;
  lb.w00 = (2 * g_lo + L - ngroups + 1) * b + 1;
  return lb;
}

// Levels L0 .. L0 + nL - 1 in one grid: block x is block j of level L (levels in order), and its W
// goes to W + (blocks of the earlier levels of the range + j) 2b b.
template <class T>
__global__ void __launch_bounds__(256) k_wy_level(int n, int b, int L0, int nL, int ngroups, int ntask,
                                                  const T* V2, const T* tau2, T* W) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int tid = threadIdx.x;
  int j = blockIdx.x, L = L0, before = 0;
  LevelBlocks lb = level_blocks(n, b, L, ngroups, ntask);
  while (j >= lb.nblk && L < L0 + nL - 1) {
    j -= lb.nblk;
    before += lb.nblk;
    ++L;
    lb = level_blocks(n, b, L, ngroups, ntask);
  }
  if (j >= lb.nblk) return;
  const int g_lo = lb.g_lo, w00 = lb.w00;
  W += (size_t)before * 2 * b * b;
  const int g = g_lo + j, t = L - (ngroups - 1 - g);
  const int m = 2 * b, ldv = m + 1;     // padded: column q of V starts q (2b + 1) elements in
  T* Vs = reinterpret_cast<T*>(smraw);  // 2b x b (ld 2b + 1)
  T* Gs = Vs + (size_t)ldv * b;         // b x b Gram V^H V, then overwritten by T (strict upper part)
  T* taus = Gs + (size_t)b * (b + 1);   // b
  const int ldg = b + 1;
  const int w0 = w00 + m * j;
  for (int idx = tid; idx < m * b; idx += blockDim.x) {
    const int r = idx % m, q = idx / m;
    const int sw = g * b + q, rel = r - q;
    T v = zero_<T>();
    if (sw <= n - 3 && rel >= 0 && rel < b && w0 + r < n) {
      const long long rid = (long long)sw * ntask + t;
      if (tau2[rid] != zero_<T>()) v = V2[rid * b + rel];
    }
    Vs[r + q * ldv] = v;
  }
  for (int q = tid; q < b; q += blockDim.x) {
    const int sw = g * b + q;
    taus[q] = (sw <= n - 3) ? tau2[(long long)sw * ntask + t] : zero_<T>();
  }
  __syncthreads();
  // Gram entries G(p, q) = v_p^H v_q, p < q (rows q .. p + b - 1 overlap)
  for (int idx = tid; idx < b * b; idx += blockDim.x) {
    const int p = idx % b, q = idx / b;
    if (p < q) {
      T acc = zero_<T>();
      for (int r = q; r < p + b; ++r) acc += cmul(Vs[r + p * ldv], Vs[r + q * ldv]);
      Gs[p + q * ldg] = acc;
    }
  }
  __syncthreads();
  // T by columns, in place over the Gram matrix's strict upper part: column q needs G(0:q, q) and the
  // finished columns 0 .. q-1 of T (diagonal: tau); one warp, two entries per lane (b <= 64)
  if (tid < 32) {
    for (int q = 0; q < b; ++q) {
      const T tq = taus[q];
      T out[2];
      for (int h = 0; h < 2; ++h) {
        const int p = tid + 32 * h;
        out[h] = zero_<T>();
        if (p < q) {
          T acc = zero_<T>();
          for (int l = p; l < q; ++l) acc += ((l == p) ? taus[p] : Gs[p + l * ldg]) * Gs[l + q * ldg];
          out[h] = -(tq * acc);
        }
      }
      __syncwarp();
      for (int h = 0; h < 2; ++h) {
        const int p = tid + 32 * h;
        if (p < q) Gs[p + q * ldg] = out[h];
      }
      __syncwarp();
    }
  }
  __syncthreads();
  // W = V T: W(r, q) = sum_{p <= q} V(r, p) T(p, q), V(r, p) != 0 for r - b < p <= r (T_pp = tau_p)
  T* Wj = W + (size_t)j * m * b;
  for (int idx = tid; idx < m * b; idx += blockDim.x) {
    const int r = idx % m, q = idx / m;
    const int p0 = max(0, r - b + 1), p1 = min(q, r);
    T acc = zero_<T>();
    for (int p = p0; p <= p1; ++p) acc += Vs[r + p * ldv] * ((p == q) ? taus[q] : Gs[p + q * ldg]);
    Wj[idx] = acc;
  }
}

// threads of a bulge-chasing block: four per output of the three products (two at b = 64)
constexpr int bulge_threads(int b) { return b == 16 ? 192 : 384; }
template <class T> size_t bulge_smem(int b) {
  return sizeof(T) * ((size_t)3 * b * (b + 1) + 7 * b + bulge_threads(b)) + 64;
}

// One cooperative launch of the chase at band width B.
template <class T, int B> int launch_bulge(Sys& s, int n, T* band, int ldb) {
  constexpr int NTH = bulge_threads(B);
  const size_t smem = bulge_smem<T>(B);
  GEV_TRY(allow_max_dyn_smem(k_bulge<T, B, NTH>));
  int per_sm = 0;
  GEV_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_bulge<T, B, NTH>, NTH + 32, smem));
  if (per_sm < 1) return GEV_ERR_UNSUPPORTED;
  // Sweep s+1 trails sweep s by a little over two tasks and a sweep runs (n - s) / b tasks, so at most
  // about n / (2b) sweeps are in flight: more blocks would only hold SMs (in a spin wait) that other
  // streams' work - concurrent solves of the serving form - could use.  Blocks that share an SM share its
  // FP64 pipe, and the pipeline runs at its slowest block's pace: a second block per SM only pays when
  // the sweeps in flight well exceed the SMs.
  int G = n / (2 * B) + 8;
  if (G > s.sms) G = 2 * G < 3 * s.sms ? s.sms : std::min(G, std::min(per_sm, 2) * s.sms);
  if (G > n - 2) G = n - 2;
  int nn = n, lb = ldb, nt = s.ntask, stall = s.opts.debug_stall ? 1 : 0;
  T* V2 = (T*)s.V2;
  T* tau2 = (T*)s.tau2;
  int* prog = s.prog;
  int* st = s.status;
  int* ab = &s.status[ST_ABORT];
  void* args[] = {&nn, &band, &lb, &V2, &tau2, &nt, &prog, &st, &ab, &stall};
  GEV_COUNT(s);
  GEV_CUDA_TRY(cudaLaunchCooperativeKernel((void*)k_bulge<T, B, NTH>, dim3(G), dim3(NTH + 32), args, smem, s.stream));
  return 0;
}

}  // namespace

template <class T> int hb2st(Sys& s, double* d, double* e) {
  const int n = s.n, b = s.band_b_used;
  const int ldb = 2 * b;
  T* band = (T*)s.band;
  if (n <= 2) {
    // already tridiagonal
  } else {
    GEV_CUDA_TRY(cudaMemsetAsync(s.prog, 0, sizeof(int) * (size_t)n, s.stream));
    GEV_CUDA_TRY(cudaMemsetAsync(s.tau2, 0, s.es() * (size_t)n * s.ntask, s.stream));
    // The FP32 back-transform applies every stored slot with its tau (no branch), so the slots of
    // tasks that never ran (a sweep ends without storing a reflector for its last single row) must
    // hold zeros, not whatever the workspace held before: 0 * NaN would poison the column.
    if constexpr (std::is_same<T, float>::value)
      GEV_CUDA_TRY(cudaMemsetAsync(s.V2, 0, sizeof(T) * (size_t)b * n * s.ntask, s.stream));
    GEV_CUDA_TRY(cudaMemsetAsync(&s.status[ST_ABORT], 0, sizeof(int), s.stream));
    if (b == 16) GEV_TRY((launch_bulge<T, 16>(s, n, band, ldb)));
    else if (b == 32) GEV_TRY((launch_bulge<T, 32>(s, n, band, ldb)));
    else if (b == 64) GEV_TRY((launch_bulge<T, 64>(s, n, band, ldb)));
    else return GEV_ERR_UNSUPPORTED;
  }
  GEV_COUNT(s);
  k_tridiag_out<T><<<1, 1024, 0, s.stream>>>(n, band, ldb, d, e, (zd*)s.phase);
  GEV_TRY(last_error());
  s.have_tridiag_refl = true;
  return 0;
}

// Y <- Q2 Y, one launch of k_bt_level per level
template <class T, int B> int bt_levels(Sys& s, int n, int k, T* Y, int ldy) {
  const int ngroups = (n - 3) / B + 1;
  const size_t smem = sizeof(T) * ((size_t)B * (B + 8) + B);
  GEV_TRY(allow_dyn_smem(k_bt_level<T, B>, smem));
  const int nlevels = ngroups + s.ntask;
  for (int L = 0; L < nlevels; ++L) {
    const int nblk = level_blocks(n, B, L, ngroups, s.ntask).nblk;
    if (nblk == 0) continue;
    // 16 columns per block until the blocks fill the GPU several times over, then more
    const unsigned yb = std::min<unsigned>(cdiv(k, BTL_COLS), std::max<unsigned>(1, 12u * s.sms / nblk));
    GEV_COUNT(s);
    k_bt_level<T, B><<<dim3(nblk, yb), 8 * BTL_COLS, smem, s.stream>>>(
        n, k, L, ngroups, (const T*)s.V2, (const T*)s.tau2, s.ntask, Y, ldy);
  }
  return last_error();
}

// Y <- Q2 Y with every level applied as  P = blockdiag(V_j^H) Y_L,  Y_L -= blockdiag(V_j T_j) P  on the
// emulated FP64 product engine (Y_L: the level's rows).  Returns GEV_ERR_UNSUPPORTED, before
// launching anything, when the handle's scratch cannot hold a level's product.
template <class T> int bt_levels_wy(Sys& s, int n, int k, int b, T* Y, int ldy) {
  constexpr int cx = is_cx<T>::value ? 1 : 0;
  const int ngroups = (n - 3) / b + 1;
  const int nlevels = ngroups + s.ntask;
  T* P = (T*)s.W1;  // (nblk b) x k products V^H Y (W1 is free during the back-transform)
  T* Wb = (T*)s.Q;  // the W_j blocks of several consecutive levels (Q is free once the divide and conquer is done)
  size_t need = 0;
  int max_nblk = 0;
  for (int L = 0; L < nlevels; ++L) {
    const LevelBlocks lb = level_blocks(n, b, L, ngroups, s.ntask);
    if (lb.nblk == 0) continue;
    max_nblk = std::max(max_nblk, lb.nblk);
    const int rows = std::min(lb.nblk * 2 * b, n - lb.w00);
    need = std::max(need, gemm_f64_bdiag_scratch(lb.nblk * b, k, rows, b, 2 * b, cx));
    need = std::max(need, gemm_f64_bdiag_scratch(rows, k, lb.nblk * b, 2 * b, b, cx));
  }
  // levels whose W_j are formed in one launch: as many as the buffer holds
  const size_t per_level = (size_t)std::max(max_nblk, 1) * 2 * b * b * sizeof(T);
  const int LCHUNK = (int)std::min<size_t>(16, (size_t)n * n * sizeof(double) / per_level);
  if (need > s.ozws_bytes || (size_t)max_nblk * b * k * sizeof(T) > (size_t)n * n * sizeof(T) || LCHUNK < 1)
    return GEV_ERR_UNSUPPORTED;
  const size_t smem = sizeof(T) * ((size_t)(2 * b + 1) * b + (size_t)b * (b + 1) + b) + 64;
  GEV_TRY(allow_dyn_smem(k_wy_level<T>, smem));
  size_t woff = 0;  // offset of level L's blocks in Wb (elements)
  for (int L = 0; L < nlevels; ++L) {
    if (L % LCHUNK == 0) {  // the compact-WY blocks of the next LCHUNK levels, in one grid
      int nb = 0;
      for (int l = L; l < std::min(nlevels, L + LCHUNK); ++l) nb += level_blocks(n, b, l, ngroups, s.ntask).nblk;
      if (nb > 0) {
        GEV_COUNT(s);
        k_wy_level<T><<<nb, 256, smem, s.stream>>>(n, b, L, std::min(LCHUNK, nlevels - L), ngroups, s.ntask,
                                                   (const T*)s.V2, (const T*)s.tau2, Wb);
      }
      woff = 0;
    }
    const LevelBlocks lb = level_blocks(n, b, L, ngroups, s.ntask);
    if (lb.nblk == 0) continue;
    const int rows = std::min(lb.nblk * 2 * b, n - lb.w00);
    T* Wl = Wb + woff;
    woff += (size_t)lb.nblk * 2 * b * b;
    BdOp a1{1, cx, b, n, s.ntask, lb.g_lo, L, ngroups, lb.nblk, lb.w00, s.V2, s.tau2, nullptr};
    T* Yl = Y + lb.w00;
    const int M1 = lb.nblk * b;
    BdOp a2{2, cx, b, n, s.ntask, lb.g_lo, L, ngroups, lb.nblk, lb.w00, nullptr, nullptr, Wl};
    // From orthonormal Z (s.z_unit), Y's columns stay unit vectors under the orthogonal transforms
    // (|y_ij| <= 1), and |P_qj| = |v_q^H y_j| <= ||v_q|| <= sqrt(2) (a Householder vector with
    // v(0) = 1): both below 2, so their scales need no pass over the data
    const bool u = s.z_unit;
    if (u && gemm_f64_bdiag_level(s, M1, rows, k, a1, a2, b, Yl, ldy, P, M1)) continue;
    if (!gemm_f64_bdiag(s, M1, k, rows, a1, b, 2 * b, Yl, ldy, 1.0, 0.0, P, M1, u)) return GEV_ERR_CUDA;
    if (!gemm_f64_bdiag(s, rows, k, M1, a2, 2 * b, b, P, M1, -1.0, 1.0, Yl, ldy, u)) return GEV_ERR_CUDA;
  }
  return last_error();
}

template <int B> int bt_levels_f32(Sys& s, int n, int k, float* Y, int ldy) {
  const int ngroups = (n - 3) / B + 1;
  const size_t smem = sizeof(float) * ((size_t)2 * B * (BTF_COLS + 1) + (size_t)B * B + B) + 64;
  GEV_TRY(allow_max_dyn_smem(k_bt_level_f32<B>));
  const int nlevels = ngroups + s.ntask;
  const unsigned ycb = cdiv(k, BTF_COLS);
  for (int L = 0; L < nlevels; ++L) {
    const int gmin = ngroups - 1 - L > 0 ? ngroups - 1 - L : 0;
    GEV_COUNT(s);
    k_bt_level_f32<B><<<dim3(ngroups - gmin, ycb), BTF_COLS, smem, s.stream>>>(
        n, k, L, ngroups, (const float*)s.V2, (const float*)s.tau2, s.ntask, Y, ldy);
  }
  return last_error();
}

// Y (n x k) = Q2 D Z for real Z.
template <class T> int bt_hb2st(Sys& s, const double* Z, int ldz, int k, T* Y, int ldy) {
  const int n = s.n, b = s.band_b_used;
  {
    long long total = (long long)n * k;
    unsigned blocks = cdiv(total, 256);
    if (blocks > 16u * s.sms) blocks = 16u * s.sms;
    GEV_COUNT(s);
    k_phase_rows<T><<<blocks, 256, 0, s.stream>>>(n, k, Z, ldz, (const zd*)s.phase, Y, ldy);
    GEV_TRY(last_error());
  }
  if (n <= 2) return 0;
  if constexpr (std::is_same<T, float>::value) {
    // (block-diagonal BF16x6 products on the tensor cores measured slower than this register kernel at n = 16384: 747 ms
    // against 556 ms, their split passes and short-K products being latency bound)
    if (b == 16) return bt_levels_f32<16>(s, n, k, Y, ldy);
    if (b == 32) return bt_levels_f32<32>(s, n, k, Y, ldy);
    if (b == 64) return bt_levels_f32<64>(s, n, k, Y, ldy);
  }
  // FP64 data with the emulated product engine: each level as two block-diagonal tensor-core
  // products of its compact-WY blocks, unless the level is short: four launches against one.  Back-transform 2, ms, tensor
  // cores / reflector by reflector, at n k b (complex: 4 n k b): real b = 32 16M 4.0 / 2.9, 24M 6.1 / 5.5, 30M 6.1 / 6.5,
  // 38M 6.2 / 7.6; b = 16 12M 11.7 / 7.5, 24M 12.6 / 13.5; b = 64 19M 2.6 / 2.2, 32M 2.6 / 2.8; complex b = 16 20M 6.6 / 5.5,
  // 41M 7.0 / 9.4; b = 32 20M 4.2 / 3.5, 41M 4.3 / 4.6.
  constexpr double kBtNative = 2.6e7;
  if constexpr (std::is_same<T, double>::value || std::is_same<T, zd>::value) {
    const double fma = (double)n * k * b * (is_cx<T>::value ? 4 : 1);  // of a level, on the FP64 pipe
    if (s.emu_fp64 && fma >= kBtNative) {
      const int r = bt_levels_wy<T>(s, n, k, b, Y, ldy);
      if (r != GEV_ERR_UNSUPPORTED) return r;  // else: the scratch is too small, take the level kernel
    }
  }
  if constexpr (!std::is_same<T, float>::value) {
    if (b == 16) return bt_levels<T, 16>(s, n, k, Y, ldy);
    if (b == 32) return bt_levels<T, 32>(s, n, k, Y, ldy);
    if (b == 64) return bt_levels<T, 64>(s, n, k, Y, ldy);
  }
  return GEV_ERR_UNSUPPORTED;
}

template int hb2st<double>(Sys&, double*, double*);
template int hb2st<float>(Sys&, double*, double*);
template int bt_hb2st<float>(Sys&, const double*, int, int, float*, int);
template int hb2st<zd>(Sys&, double*, double*);
template int bt_hb2st<double>(Sys&, const double*, int, int, double*, int);
template int bt_hb2st<zd>(Sys&, const double*, int, int, zd*, int);
template int hb2st<zf>(Sys&, double*, double*);
template int bt_hb2st<zf>(Sys&, const double*, int, int, zf*, int);

}  // namespace gev
