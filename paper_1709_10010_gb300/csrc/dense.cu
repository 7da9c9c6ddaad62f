// Small dense FP64 linear algebra on the device for the Davidson subspace
// (the O_ij = <psi_i|O|psi_j> matrices and their "subspace diagonalization",
// Sec. "New parallelization levels"):
//
//  * jacobi_eigh   Hermitian eigensolver, cyclic parallel (round-robin pairing)
//                  two-sided Jacobi with complex rotations; one cooperative
//                  launch, rounds separated by a bounded grid barrier.
//  * cholqr_factor Cholesky of a Gram matrix with column dropping, returning the
//                  k x k' transform Tr with T Tr orthonormal.
//  * hermitize     completes and symmetrises freshly computed columns of the
//                  subspace matrix.
//
// Every spin in these kernels is bounded (about one second of %globaltimer);
// a kernel that gives up records PWH_ERR_TIMEOUT in the device error word and
// returns.
#include <algorithm>
#include <cmath>
#include <map>
#include <mutex>

#include "common.cuh"
#include "dense.cuh"
#include "gemm.cuh"
#include "jacobi_rot.cuh"

namespace pwh {

constexpr unsigned long long kWaitNs = 1000000000ull;

__device__ __forceinline__ uint64_t gtimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier for a cooperative launch (all blocks resident).  One arrival
// counter, zeroed before the launch and never reset inside it: the e-th
// barrier of a block (its own epoch count; every block passes the same
// barriers) is complete once the counter reaches e * gridDim.x.  Thread 0
// arrives with a release-acquire add (publishing the block's writes, ordered
// before it by the first __syncthreads) and polls with acquire loads, so the
// whole block sees every other block's writes after the second
// __syncthreads.  Returns false (after recording the error) if the wait ran
// out or another block already gave up.
struct GridBar {
  unsigned* count;
  unsigned* unused;
  int* abort;
  int* err;
};

__device__ __forceinline__ unsigned atom_add_acq_rel_gpu(unsigned* p, unsigned v) {
  unsigned old;
  asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], %2;" : "=r"(old) : "l"(p), "r"(v) : "memory");
  return old;
}
__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ bool grid_sync(const GridBar& gb, unsigned& epoch) {
  __shared__ int s_ok;
  __syncthreads();
  ++epoch;
  if (threadIdx.x == 0) {
    int ok = 1;
    const unsigned target = epoch * gridDim.x;
    unsigned v = atom_add_acq_rel_gpu(gb.count, 1u) + 1u;
    if ((int)(v - target) < 0) {
      const uint64_t t0 = gtimer_ns();
      unsigned it = 0;
      while ((int)(ld_acquire_gpu(gb.count) - target) < 0) {
        if ((++it & 63) == 0) {
          if (*(volatile int*)gb.abort) {
            ok = 0;
            break;
          }
          if (gtimer_ns() - t0 > kWaitNs) {
            ok = 0;
            atomicExch(gb.abort, 1);
            atomicExch(gb.err, (int)PWH_ERR_TIMEOUT);
            break;
          }
        }
      }
    }
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Index at tournament position j in round r of a round-robin over n (even)
// players: position 0 fixed, the others rotate.
__device__ __forceinline__ int rr_player(int j, int r, int n) {
  return j == 0 ? 0 : 1 + ((j - 1 + r) % (n - 1));
}

__device__ __forceinline__ double cabs2(double2 z) { return z.x * z.x + z.y * z.y; }

// Parallel cyclic Jacobi on A (n x n Hermitian, column-major ld = n; ping-pong
// buffers A[0]/A[1], Q[0]/Q[1]; A[0] holds the start and Q[0] the basis it is
// expressed in).  n is padded to even np with a dummy index that never
// rotates.  In round r of the round-robin the np/2 disjoint pairs (p, q) each
// get the rotation J = [[c, s], [-conj(s), c]] (c real, s = |s| e^{i phi})
// that zeroes A_pq, and A' = J^H A J, Q' = Q J are formed in one pass: a work
// item is a 2 x 2 block of A (rows of pair k, columns of pair l, k <= l by
// Hermitian symmetry; the mirror block is written too) or one row of Q
// against one pair.  Every block recomputes the round's rotations in shared
// memory, so a round costs one grid barrier.  After each sweep block 0 scans
// the off-diagonal of the current A; the sweeps stop in lockstep once
// max|A_ij| <= tol * max|A_ii|.
template <typename T>
struct JacobiArgsT {
  cx<T>* A[2];
  cx<T>* Q[2];
  int n, np, max_sweeps;
  double tol;
  int* out_buf;   // buffer index (0/1) holding the result, sweeps used
  int* conv;      // per-sweep convergence flag written by block 0
  // of a polish (KEEP), else null.  skip: nonzero = already diagonal, no sweep;
  // dmax: max |A_ii|, pairs with |A_pq| <= 1e-15 of it keep their element and are not
  // rotated
  const int* skip;
  const unsigned long long* dmax;
  GridBar gb;
};

// All threads of all CTAs of the cluster (the whole grid when launched as one
// cluster): hardware barrier with release/acquire ordering at cluster scope.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile(
      "barrier.cluster.arrive.release.aligned;\n"
      "barrier.cluster.wait.acquire.aligned;\n" ::: "memory");
}

// CLUSTER: the grid is one thread-block cluster and rounds are separated by
// the hardware cluster barrier; otherwise by the bounded grid barrier of a
// cooperative launch.
// KEEP (FP64): the polish of an almost diagonal matrix, with a.dmax.
template <typename T, bool CLUSTER, bool KEEP = false>
__global__ void k_jacobi(JacobiArgsT<T> a) {
  extern __shared__ __align__(16) unsigned char jsm[];
  const int n = a.n, np = a.np, P = np / 2;
  cx<T>* srot = (cx<T>*)jsm;          // P: s of pair k
  T* crot = (T*)(srot + P);           // P: c of pair k
  int* pp = (int*)(crot + P);         // P: p of pair k
  int* pq = pp + P;                   // P: q of pair k
  __shared__ double s_red[2][32];
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int nth = gridDim.x * blockDim.x;
  unsigned epoch = 0;  // grid barriers passed
  int cur = 0, sweep = 0;
  const int max_sweeps = KEEP && *a.skip ? 0 : a.max_sweeps;
  double keep2 = -1.0;  // |A_pq|^2 up to which a pair is left alone
  if constexpr (KEEP) {
    const double d = 1e-15 * __longlong_as_double((long long)*a.dmax);
    keep2 = d * d;
  }
  for (; sweep < max_sweeps; ++sweep) {
    for (int r = 0; r < np - 1; ++r) {
      const cx<T>* A = a.A[cur];
      for (int k = threadIdx.x; k < P; k += blockDim.x) {
        int p = rr_player(k, r, np), q = rr_player(np - 1 - k, r, np);
        if (p > q) { int t = p; p = q; q = t; }
        T c = 1;
        cx<T> sv = mk<T>(0, 0);
        if (q < n) {
          const cx<T> apq = A[(size_t)q * n + p];
          if (!KEEP || !((double)apq.x * apq.x + (double)apq.y * apq.y <= keep2))
            jacobi_rotation<T>(apq, A[(size_t)p * n + p].x, A[(size_t)q * n + q].x, c, sv);
        }
        pp[k] = p;
        pq[k] = q;
        crot[k] = c;
        srot[k] = sv;
      }
      __syncthreads();
      const cx<T>* Qc = a.Q[cur];
      cx<T>* An = a.A[cur ^ 1];
      cx<T>* Qn = a.Q[cur ^ 1];
      const int nA = P * P, nQ = n * P;
      for (int t = tid; t < nA + nQ; t += nth) {
        if (t < nA) {
          const int k = t % P, l = t / P;
          if (k > l) continue;
          const int pk = pp[k], qk = pq[k], pl = pp[l], ql = pq[l];
          const bool vk = qk < n, vl = ql < n;  // pair carries a real second index
          if (pk >= n || pl >= n) continue;     // (p is never the dummy: p < q)
          const T ck = crot[k], cl = crot[l];
          const cx<T> sk = srot[k], sl = srot[l];
          const cx<T> z = mk<T>(0, 0);
          const cx<T> a00 = A[(size_t)pl * n + pk];
          const cx<T> a01 = vl ? A[(size_t)ql * n + pk] : z;
          const cx<T> a10 = vk ? A[(size_t)pl * n + qk] : z;
          const cx<T> a11 = (vk && vl) ? A[(size_t)ql * n + qk] : z;
          cx<T> y00, y01, y10, y11;
          // neither pair rotates (the polish of an almost diagonal matrix):
          // the block moves to the other buffer without FP64 arithmetic
          const bool still = KEEP && ck == (T)1 && cl == (T)1 &&
                             sk.x == (T)0 && sk.y == (T)0 && sl.x == (T)0 && sl.y == (T)0;
          if (still) {
            y00 = a00; y01 = a01; y10 = a10; y11 = a11;
          } else {
            jacobi_block<T>(a00, a01, a10, a11, ck, sk, cl, sl, y00, y01, y10, y11);
          }
          if (k == l && !still) {
            // rotated 2 x 2 diagonal block: real diagonal, zeroed pair element
            An[(size_t)pk * n + pk] = mk<T>(y00.x, 0);
            if (vk) {
              An[(size_t)qk * n + qk] = mk<T>(y11.x, 0);
              An[(size_t)qk * n + pk] = mk<T>(0, 0);
              An[(size_t)pk * n + qk] = mk<T>(0, 0);
            }
          } else {
            An[(size_t)pl * n + pk] = y00;
            An[(size_t)pk * n + pl] = mk<T>(y00.x, -y00.y);
            if (vl) {
              An[(size_t)ql * n + pk] = y01;
              An[(size_t)pk * n + ql] = mk<T>(y01.x, -y01.y);
            }
            if (vk) {
              An[(size_t)pl * n + qk] = y10;
              An[(size_t)qk * n + pl] = mk<T>(y10.x, -y10.y);
            }
            if (vk && vl) {
              An[(size_t)ql * n + qk] = y11;
              An[(size_t)qk * n + ql] = mk<T>(y11.x, -y11.y);
            }
          }
        } else {
          const int e = t - nA;
          const int i = e % n, l = e / n;
          const int pl = pp[l], ql = pq[l];
          if (pl >= n) continue;
          const T cl = crot[l];
          const cx<T> sl = srot[l];
          const cx<T> q0 = Qc[(size_t)pl * n + i];
          if (KEEP && ql < n && cl == (T)1 && sl.x == (T)0 && sl.y == (T)0) {
            Qn[(size_t)pl * n + i] = q0;
            Qn[(size_t)ql * n + i] = Qc[(size_t)ql * n + i];
          } else if (ql < n) {
            const cx<T> q1 = Qc[(size_t)ql * n + i];
            Qn[(size_t)pl * n + i] = add<T>(scl<T>(q0, cl), mul<T>(q1, mk<T>(-sl.x, sl.y)));
            Qn[(size_t)ql * n + i] = add<T>(mul<T>(q0, sl), scl<T>(q1, cl));
          } else {
            Qn[(size_t)pl * n + i] = q0;
          }
        }
      }
      cur ^= 1;
      if (CLUSTER) {
        cluster_sync_all();
      } else if (!grid_sync(a.gb, epoch)) {
        return;
      }
    }
    // convergence of the current matrix, decided by block 0 for everyone
    if (blockIdx.x == 0) {
      const cx<T>* A = a.A[cur];
      double off = 0.0, dm = 0.0;
      for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
        const int i = t % n, j = t / n;
        const cx<T> v = A[t];
        if (i == j) dm = fmax(dm, fabs((double)v.x));
        else if (i < j) off = fmax(off, sqrt((double)v.x * v.x + (double)v.y * v.y));
      }
      for (int o = 16; o > 0; o >>= 1) {
        off = fmax(off, __shfl_xor_sync(0xffffffffu, off, o));
        dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
      }
      if ((threadIdx.x & 31) == 0) {
        s_red[0][threadIdx.x >> 5] = off;
        s_red[1][threadIdx.x >> 5] = dm;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
          s_red[0][0] = fmax(s_red[0][0], s_red[0][w]);
          s_red[1][0] = fmax(s_red[1][0], s_red[1][w]);
        }
        *(volatile int*)a.conv = s_red[0][0] <= a.tol * fmax(s_red[1][0], 1e-300) ? 1 : 0;
      }
    }
    if (CLUSTER) {
      cluster_sync_all();
    } else if (!grid_sync(a.gb, epoch)) {
      return;
    }
    if (*(volatile int*)a.conv) {
      ++sweep;
      break;
    }
  }
  if (tid == 0) {
    a.out_buf[0] = cur;
    a.out_buf[1] = sweep;
  }
}

// dst (FP64) = the FP32 buffer (b0 or b1) holding the result.
__global__ void k_select_buf(const float2* __restrict__ b0, const float2* __restrict__ b1,
                             const int* __restrict__ buf, int64_t n2, double2* __restrict__ dst) {
  const float2* b = buf[0] ? b1 : b0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n2;
       t += (int64_t)gridDim.x * blockDim.x)
    dst[t] = make_double2((double)b[t].x, (double)b[t].y);
}

// Lowest nk eigenpairs from a diagonal d (n) and eigenvector matrix Q (n x n,
// ld n): theta[rank], C[:, rank] for rank < nk, and every column into Qkeep
// (ld ldk) in ascending order.  Ties go to the lower index.  Each block ranks
// all n values itself (n^2 comparisons) and copies a slice of the columns.
__global__ void k_select_eig(const double* __restrict__ d, const double2* __restrict__ Q, int n,
                             int nk, double* __restrict__ theta, double2* __restrict__ C,
                             double2* __restrict__ Qkeep, int64_t ldk) {
  extern __shared__ int rank_of[];
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double di = d[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      const double dj = d[j];
      rank += (dj < di) || (dj == di && j < i);
    }
    rank_of[i] = rank;
    if (blockIdx.x == 0 && rank < nk) theta[rank] = di;
  }
  __syncthreads();
  const int64_t tot = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t / n), r = (int)(t - (int64_t)i * n);
    const int rank = rank_of[i];
    const double2 v = Q[t];
    if (rank < nk) C[(size_t)rank * n + r] = v;
    if (Qkeep) Qkeep[(size_t)rank * ldk + r] = v;
  }
}

// d[i] = Re(Q[:, i]^H G[:, i]) (G = H Q): Rayleigh quotients, one block per column.
__global__ void k_rayleigh(const double2* __restrict__ Q, const double2* __restrict__ G, int n,
                           double* __restrict__ d) {
  __shared__ double part[32];
  const int i = blockIdx.x;
  double acc = 0.0;
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    const double2 q = Q[(size_t)i * n + r], g = G[(size_t)i * n + r];
    acc += q.x * g.x + q.y * g.y;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += part[w];
    d[i] = t;
  }
}

// d = diagonal of the n x n matrix held in a0 or a1 (buf[0]), either precision.
template <typename T>
__global__ void k_diag_of(const cx<T>* __restrict__ a0, const cx<T>* __restrict__ a1,
                          const int* __restrict__ buf, int n, double* __restrict__ d) {
  const cx<T>* a = (buf && buf[0]) ? a1 : a0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    d[i] = (double)a[(size_t)i * n + i].x;
}

// dst = the FP64 buffer (b0 or b1) holding the result.
__global__ void k_select_buf64(const double2* __restrict__ b0, const double2* __restrict__ b1,
                               const int* __restrict__ buf, int64_t n2, double2* __restrict__ dst) {
  const double2* b = buf[0] ? b1 : b0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n2;
       t += (int64_t)gridDim.x * blockDim.x)
    dst[t] = b[t];
}

// Q0 = blockdiag(Qprev[0:m0, 0:m0], I) (n x n, ld n).
__global__ void k_warm_basis(const double2* __restrict__ Qprev, int64_t ldp, int m0, int n,
                             double2* __restrict__ Q0) {
  int64_t tot = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(t % n), j = (int)(t / n);
    double2 v = make_double2(i == j ? 1.0 : 0.0, 0.0);
    if (i < m0 && j < m0) v = Qprev[(size_t)j * ldp + i];
    else if (i < m0 || j < m0) v = make_double2(0.0, 0.0);
    Q0[t] = v;
  }
}

// Complete columns [m0, m) of the Hermitian subspace matrix H (ld): rows
// [0, m0) mirror into the lower-left block; the new diagonal block is
// replaced by its Hermitian part.
__global__ void k_hermitize(double2* __restrict__ H, int64_t ld, int m0, int m) {
  const int k = m - m0;
  int64_t tot = (int64_t)m * k;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(t % m), j = m0 + (int)(t / m);
    if (i < m0) {
      double2 z = H[(size_t)j * ld + i];
      H[(size_t)i * ld + j] = make_double2(z.x, -z.y);
    } else if (i < j) {
      double2 a = H[(size_t)j * ld + i], b = H[(size_t)i * ld + j];
      double2 av = make_double2(0.5 * (a.x + b.x), 0.5 * (a.y - b.y));
      H[(size_t)j * ld + i] = av;
      H[(size_t)i * ld + j] = make_double2(av.x, -av.y);
    } else if (i == j) {
      H[(size_t)j * ld + i].y = 0.0;
    }
  }
}

// Cholesky-QR factor of a Gram matrix S = T^H T (k x k, ld = k), one block.
// Column j survives when S_jj > 0, sqrt(S_jj) >= drop_rel * t0[j] (t0 may be
// null) and its Cholesky pivot of the unit-diagonal matrix stays above
// piv_tol.  Output: Tr (k x k, ld = k) whose first kk columns give T Tr with
// orthonormal columns (other columns zero); *kk = number kept.  The lower
// triangle lives in shared memory (packed by columns) when SMEM, else in the
// k x k global scratch W.
template <typename T, bool SMEM>
__global__ void __launch_bounds__(1024) k_cholqr(const double2* __restrict__ S, int k,
                                                 const double* __restrict__ t0, double drop_rel,
                                                 double piv_tol, cx<T>* __restrict__ Wg,
                                                 double2* __restrict__ Tr, int* __restrict__ kk) {
  extern __shared__ __align__(16) unsigned char chsm[];
  __shared__ int keep_s[1024];
  __shared__ int rank_s[1024];
  __shared__ double dinv_s[1024];
  __shared__ int nkeep_s;
  __shared__ T piv_s;
  cx<T>* L = SMEM ? (cx<T>*)chsm : Wg;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  // element (i, j), i >= j, of the lower triangle (packed by columns in
  // shared memory, else a k x k column-major scratch)
  auto at = [&](int i, int j) -> cx<T>& {
    return SMEM ? L[(size_t)j * k - (size_t)j * (j - 1) / 2 + (i - j)] : L[(size_t)j * k + i];
  };
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    double d = S[(size_t)j * k + j].x;
    bool keep = d > 0.0 && (!t0 || sqrt(d) >= drop_rel * t0[j]);
    keep_s[j] = keep;
    dinv_s[j] = keep ? 1.0 / sqrt(d) : 0.0;
  }
  __syncthreads();
  // unit-diagonal scaling of the lower triangle (a warp per column)
  for (int j = warp; j < k; j += nwarps)
    for (int i = j + lane; i < k; i += 32) {
      const double2 v = S[(size_t)j * k + i];
      const double sc = dinv_s[i] * dinv_s[j];
      at(i, j) = mk<T>((T)(v.x * sc), (T)(v.y * sc));
    }
  __syncthreads();
  // right-looking Cholesky on the kept set
  for (int j = 0; j < k; ++j) {
    if (threadIdx.x == 0) {
      const T piv = at(j, j).x;
      if (keep_s[j] && !(piv > (T)piv_tol)) keep_s[j] = 0;
      piv_s = keep_s[j] ? sqrt(piv) : (T)0;
    }
    __syncthreads();
    if (keep_s[j]) {
      const T rl = (T)1 / piv_s;
      for (int i = j + 1 + threadIdx.x; i < k; i += blockDim.x)
        if (keep_s[i]) at(i, j) = scl<T>(at(i, j), rl);
      __syncthreads();
      // trailing update of the lower triangle: a warp per column l, lanes over rows i >= l
      for (int l = j + 1 + warp; l < k; l += nwarps) {
        if (!keep_s[l]) continue;
        const cx<T> ljc = at(l, j);
        for (int i = l + lane; i < k; i += 32)
          if (keep_s[i]) at(i, l) = sub<T>(at(i, l), mulc<T>(at(i, j), ljc));
      }
      if (threadIdx.x == 0) at(j, j) = mk<T>(piv_s, (T)0);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    int c = 0;
    for (int j = 0; j < k; ++j) rank_s[j] = keep_s[j] ? c++ : -1;
    nkeep_s = c;
    *kk = c;
  }
  __syncthreads();
  // L <- L^-1 in place on the kept set, columns from the last: for i > j,
  // (L^-1)_ij = -(1/L_jj) sum_{j < l <= i} (L^-1)_il L_lj, with the trailing
  // block already inverted; the original column j is kept in col_s.  A warp
  // per row i, lanes over l.
  __shared__ cx<T> col_s[1024];
  for (int j = k - 1; j >= 0; --j) {
    if (!keep_s[j]) continue;
    for (int i = j + 1 + threadIdx.x; i < k; i += blockDim.x)
      col_s[i] = keep_s[i] ? at(i, j) : mk<T>((T)0, (T)0);
    __syncthreads();
    const T djj = (T)1 / at(j, j).x;
    for (int i = j + 1 + warp; i < k; i += nwarps) {
      if (!keep_s[i]) continue;
      cx<T> acc = mk<T>((T)0, (T)0);
      for (int l = j + 1 + lane; l <= i; l += 32)
        if (keep_s[l]) acc = add<T>(acc, mul<T>(at(i, l), col_s[l]));
      for (int o = 16; o > 0; o >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, o);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, o);
      }
      if (lane == 0) at(i, j) = scl<T>(acc, -djj);
    }
    if (threadIdx.x == 0) at(j, j) = mk<T>(djj, (T)0);
    __syncthreads();
  }
  // Tr = D^-1/2 L^-H: column rank(j), row i <= j holds conj((L^-1)_ji) / sqrt(S_ii)
  for (int t = threadIdx.x; t < k * k; t += blockDim.x) Tr[t] = make_double2(0.0, 0.0);
  __syncthreads();
  for (int t = threadIdx.x; t < k * k; t += blockDim.x) {
    const int i = t % k, j = t / k;
    if (i > j || !keep_s[i] || !keep_s[j]) continue;
    const cx<T> v = at(j, i);
    Tr[(size_t)rank_s[j] * k + i] = make_double2((double)v.x * dinv_s[i], -(double)v.y * dinv_s[i]);
  }
}

// FP32 <-> FP64 copies and the Newton-Schulz step of the host routine.
__global__ void k_c64_to_c32(const double2* __restrict__ a, int64_t lda, int n, float2* __restrict__ b) {
  int64_t tot = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(t % n), j = (int)(t / n);
    double2 z = a[(size_t)j * lda + i];
    b[t] = make_float2((float)z.x, (float)z.y);
  }
}
__global__ void k_c32_to_c64(const float2* __restrict__ a, int64_t n2, double2* __restrict__ b) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n2;
       t += (int64_t)gridDim.x * blockDim.x)
    b[t] = make_double2((double)a[t].x, (double)a[t].y);
}
// B = (3 I - G) / 2
__global__ void k_ns_rhs(const double2* __restrict__ G, int n, double2* __restrict__ B) {
  int64_t tot = (int64_t)n * n;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    int i = (int)(t % n), j = (int)(t / n);
    double2 g = G[t];
    B[t] = make_double2((i == j ? 1.5 : 0.0) - 0.5 * g.x, -0.5 * g.y);
  }
}

// ---- FP32 Jacobi over the whole GPU in tournament-position order --------
// For subspaces too large for one cluster's shared memory.  The matrix is
// stored by tournament position instead of by index: pair k of every round
// is positions (2k, 2k+1), so a round reads each 2 x 2 block (rows of pair k,
// columns of pair l) as two contiguous 16-byte runs.  The circle method moves
// the players between rounds along one cycle (position 0 stays; 2 -> 4 ->
// ... -> np-2 -> np-1 -> np-3 -> ... -> 1 -> 2), and each round writes every
// rotated element straight to its position of the next round, in the other
// buffer, so the move costs no extra pass.  After np - 1 rounds every player
// is back where it started: at a sweep boundary position = index.  Blocks
// are taken in tiles of kPjTile x kPjTile pairs; only the upper triangle is
// stored: tiles on or above the diagonal are computed and each element is
// written once, at its canonical (upper) next-round position, conjugated where
// the move swapped row and column order (a round reads half the matrix and
// writes half).  The rotations go to a log in index form, (s, c, p | q << 16)
// per pair and round, from which k_jacobi_qlog_rows forms Q afterwards.
constexpr int kPjTile = 16;
constexpr int kPjGroup = kPjTile * kPjTile;  // threads on one tile
constexpr int kPjTiles = 4;                  // tiles a block works on at once
constexpr int kPjThreads = kPjGroup * kPjTiles;

// A stores its upper triangle only (position order, column-major): element
// (row, col) goes to (min, max), conjugated when the move swapped their order.
__device__ __forceinline__ void pj_store_upper(float2* A, int np, int row, int col, float2 y) {
  if (row <= col)
    A[(size_t)col * np + row] = y;
  else
    A[(size_t)row * np + col] = make_float2(y.x, -y.y);
}

// next position of the player at x (np even)
__device__ __forceinline__ int pj_next(int x, int np) {
  if (x == 0 || np == 2) return x;
  if (x == 1) return 2;
  if ((x & 1) == 0) return x == np - 2 ? np - 1 : x + 2;
  return x - 2;
}
// index standing at position x in round r (0 <= r < np - 1) of a sweep
__device__ __forceinline__ int pj_index(int x, int r, int np) {
  if (x == 0) return 0;
  const int P = np / 2, L = np - 1;
  const int c = (x & 1) ? P - 1 + (np - 1 - x) / 2 : x / 2 - 1;  // place on the cycle
  int c0 = c - r;
  if (c0 < 0) c0 += L;
  return c0 <= P - 2 ? 2 * c0 + 2 : np - 1 - 2 * (c0 - (P - 1));
}

struct PjArgs {
  float2* A[2];       // np x np, column-major, by position; A[0] holds the start
  float4* log;        // round t, pair k at [t P + k]: (s.x, s.y, c, p | q << 16)
  int64_t log_rounds;
  double* diag;       // out: final diagonal, by index
  int* info;          // out: [0] buffer of the final matrix, [1] sweeps, [2] rounds logged
  unsigned* red;      // 2 words per sweep (max off-diagonal, max diagonal; float bits), zeroed
  int n, np, P, T, max_sweeps;
  float tol;
  GridBar gb;
};

__global__ void __launch_bounds__(kPjThreads) k_jacobi_pos(PjArgs a) {
  extern __shared__ __align__(16) unsigned char pjs[];
  float4* rot = (float4*)pjs;               // P rotations (s.x, s.y, c, -)
  const int grp = threadIdx.x / kPjGroup, gt = threadIdx.x % kPjGroup;
  __shared__ float s_red[2][kPjThreads / 32];
  const int np = a.np, P = a.P, T = a.T, n = a.n;
  const int ntiles = T * (T + 1) / 2;
  const int gtid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  int cur = 0, sweep = 0, rounds = 0;
  unsigned epoch = 0;  // grid barriers passed
  bool done = false;
  while (sweep < a.max_sweeps && !done) {
    for (int r = 0; r < np - 1; ++r) {
      const float2* A = cur ? a.A[1] : a.A[0];
      float2* An = cur ? a.A[0] : a.A[1];
      const int kl = gt % kPjTile, ll = gt / kPjTile;
      // upper-triangle tile (I, J), I <= J, numbered row by row; its two
      // 16-byte loads for this thread's pair of pairs (k, l) when it has one
      auto tile_load = [&](int tile, int& I, int& J, bool& act, float4& c0, float4& c1) {
        int i = 0, rem = tile < ntiles ? tile : 0;
        while (rem >= T - i) {
          rem -= T - i;
          ++i;
        }
        I = i;
        J = i + rem;
        const int k = I * kPjTile + kl, l = J * kPjTile + ll;
        act = tile < ntiles && k < P && l < P && (I != J || kl <= ll);
        if (act) {
          c0 = *(const float4*)(A + (size_t)(2 * l) * np + 2 * k);      // a00, a10
          c1 = *(const float4*)(A + (size_t)(2 * l + 1) * np + 2 * k);  // a01, a11
        }
      };
      // the block's first tile is loaded before the rotations are formed, so
      // both L2 round trips of the round overlap
      const int stride = gridDim.x * kPjTiles;
      int t0 = blockIdx.x * kPjTiles;
      int I, J;
      bool act;
      float4 c0 = make_float4(0.f, 0.f, 0.f, 0.f), c1 = c0;
      tile_load(t0 + grp, I, J, act, c0, c1);
      for (int k = threadIdx.x; k < P; k += blockDim.x) {
        const size_t d = (size_t)(2 * k) * np + 2 * k;
        float c;
        float2 sv;
        jacobi_rotation<float>(A[d + np], A[d].x, A[d + np + 1].x, c, sv);
        rot[k] = make_float4(sv.x, sv.y, c, 0.f);
        if (blockIdx.x == 0 && rounds < a.log_rounds) {
          const int p = pj_index(2 * k, r, np), q = pj_index(2 * k + 1, r, np);
          a.log[(size_t)rounds * P + k] = make_float4(sv.x, sv.y, c, __int_as_float(p | (q << 16)));
        }
      }
      __syncthreads();
      // kPjTiles tiles at once, one per group of threads; every group runs
      // the same number of iterations (the barriers stay uniform); the next
      // tile's operands are fetched while the current one is rotated
      for (; t0 < ntiles; t0 += stride) {
        int In = 0, Jn = 0;
        bool actn = false;
        float4 n0 = c0, n1 = c1;
        if (t0 + stride < ntiles) tile_load(t0 + stride + grp, In, Jn, actn, n0, n1);
        const int k = I * kPjTile + kl, l = J * kPjTile + ll;
        if (act) {
          const float4 rk = rot[k], rl = rot[l];
          // the diagonal 2 x 2 block keeps only its upper element: a10 = conj(a01)
          const float2 a01 = make_float2(c1.x, c1.y);
          const float2 a10 = k == l ? make_float2(c1.x, -c1.y) : make_float2(c0.z, c0.w);
          float2 y00, y01, y10, y11;
          jacobi_block<float>(make_float2(c0.x, c0.y), a01, a10, make_float2(c1.z, c1.w), rk.z,
                              make_float2(rk.x, rk.y), rl.z, make_float2(rl.x, rl.y), y00, y01,
                              y10, y11);
          if (k == l) {
            // the rotated diagonal block: real diagonal, zeroed pair element
            y00.y = 0.f;
            y11.y = 0.f;
            y01 = make_float2(0.f, 0.f);
          }
          const int i0 = pj_next(2 * k, np), i1 = pj_next(2 * k + 1, np);
          const int j0 = pj_next(2 * l, np), j1 = pj_next(2 * l + 1, np);
          pj_store_upper(An, np, i0, j0, y00);
          pj_store_upper(An, np, i0, j1, y01);
          pj_store_upper(An, np, i1, j1, y11);
          if (k != l) pj_store_upper(An, np, i1, j0, y10);
        }
        I = In;
        J = Jn;
        act = actn;
        c0 = n0;
        c1 = n1;
      }
      ++rounds;
      cur ^= 1;
      if (!grid_sync(a.gb, epoch)) return;
    }
    // convergence of the current matrix (position = index again): grid-wide
    // maxima of |A_ij| (i < j) and |A_ii|, every block takes the same decision
    {
      const float2* A = cur ? a.A[1] : a.A[0];
      float off = 0.f, dm = 0.f;
      for (int64_t t = gtid; t < (int64_t)n * n; t += nth) {
        const int i = (int)(t % n), j = (int)(t / n);
        const float2 v = A[(size_t)j * np + i];
        if (i == j) dm = fmaxf(dm, fabsf(v.x));
        else if (i < j) off = fmaxf(off, sqrtf(v.x * v.x + v.y * v.y));
      }
      for (int o = 16; o > 0; o >>= 1) {
        off = fmaxf(off, __shfl_xor_sync(0xffffffffu, off, o));
        dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
      }
      if ((threadIdx.x & 31) == 0) {
        s_red[0][threadIdx.x >> 5] = off;
        s_red[1][threadIdx.x >> 5] = dm;
      }
      __syncthreads();
      if (threadIdx.x == 0) {
        for (int w = 1; w < kPjThreads / 32; ++w) {
          off = fmaxf(s_red[0][0], s_red[0][w]);
          s_red[0][0] = off;
          s_red[1][0] = fmaxf(s_red[1][0], s_red[1][w]);
        }
        atomicMax(a.red + 2 * sweep, __float_as_uint(s_red[0][0]));
        atomicMax(a.red + 2 * sweep + 1, __float_as_uint(s_red[1][0]));
      }
      if (!grid_sync(a.gb, epoch)) return;
      const float offg = __uint_as_float(*(volatile unsigned*)(a.red + 2 * sweep));
      const float dmg = __uint_as_float(*(volatile unsigned*)(a.red + 2 * sweep + 1));
      done = offg <= a.tol * fmaxf(dmg, 1e-30f);
    }
    ++sweep;
  }
  if (gtid == 0) {
    a.info[0] = cur;
    a.info[1] = sweep;
    a.info[2] = (int)min((int64_t)rounds, a.log_rounds);
  }
  const float2* Af = cur ? a.A[1] : a.A[0];
  for (int i = gtid; i < n; i += nth) a.diag[i] = (double)Af[(size_t)i * np + i].x;
}

// FP64 start (n x n, ld lda) -> FP32 np x np by position (= index), zero padded.
__global__ void k_to_pos32(const double2* __restrict__ A, int64_t lda, int n, int np,
                           float2* __restrict__ out) {
  const int64_t tot = (int64_t)np * np;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % np), j = (int)(t / np);
    const double2 z = (i < n && j < n) ? A[(size_t)j * lda + i] : make_double2(0.0, 0.0);
    out[t] = make_float2((float)z.x, (float)z.y);
  }
}

// Q = J_0 J_1 ... J_{R-1} from the log of k_jacobi_pos (R = info[2]): the rows
// of Q evolve independently, `rows` rows a block in shared memory (starting
// as rows of the identity), every round applied to them in order.  Thread t
// owns pairs t and t + blockDim (P <= 2 blockDim) and applies them to every
// row of the block; the next round's log entries are fetched before the
// barrier that closes the current round.
__global__ void __launch_bounds__(1024) k_jacobi_qlog_rows(const float4* __restrict__ log,
                                                           const int* __restrict__ info, int n,
                                                           int P, int rows, double2* __restrict__ Q,
                                                           int64_t ldq) {
  extern __shared__ __align__(16) unsigned char qrs[];
  float2* qs = (float2*)qrs;  // [rows][n]
  const int i0 = blockIdx.x * rows;
  const int nr = min(rows, n - i0);
  for (int t = threadIdx.x; t < rows * n; t += blockDim.x) {
    const int r = t / n, c = t - r * n;
    qs[t] = make_float2((r < nr && i0 + r == c) ? 1.f : 0.f, 0.f);
  }
  const int R = info[2];
  const int k0 = threadIdx.x, k1 = threadIdx.x + blockDim.x;
  const float4 idle = make_float4(0.f, 0.f, 1.f, __int_as_float(0xffff | (0xffff << 16)));
  float4 c0 = (R > 0 && k0 < P) ? log[k0] : idle, c1 = (R > 0 && k1 < P) ? log[k1] : idle;
  __syncthreads();
  for (int rd = 0; rd < R; ++rd) {
    const float4 u0 = c0, u1 = c1;
    if (rd + 1 < R) {
      const float4* nx = log + (size_t)(rd + 1) * P;
      c0 = k0 < P ? __ldg(nx + k0) : idle;
      c1 = k1 < P ? __ldg(nx + k1) : idle;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 cur = h ? u1 : u0;
      const int pq = __float_as_int(cur.w);
      const int p = pq & 0xffff, q = (pq >> 16) & 0xffff;
      if (p < n && q < n) {
        const float c = cur.z;
        const float2 sv = make_float2(cur.x, cur.y), sm = make_float2(-cur.x, cur.y);
        for (int r = 0; r < nr; ++r) {
          float2* row = qs + (size_t)r * n;
          const float2 q0 = row[p], q1 = row[q];
          row[p] = add<float>(scl<float>(q0, c), mul<float>(q1, sm));
          row[q] = add<float>(mul<float>(q0, sv), scl<float>(q1, c));
        }
      }
    }
    __syncthreads();
  }
  for (int t = threadIdx.x; t < nr * n; t += blockDim.x) {
    const int c = t / nr, rr = t - c * nr;
    const float2 v = qs[(size_t)rr * n + c];
    Q[(size_t)c * ldq + i0 + rr] = make_double2((double)v.x, (double)v.y);
  }
}

static size_t pj_log_bytes(int n, int max_sweeps) {
  const int np = n + (n & 1);
  return (size_t)max_sweeps * (np - 1) * (np / 2) * sizeof(float4) + 256;
}
static size_t pj_buf_bytes(int n) {
  const int np = n + (n & 1);
  return 2 * (size_t)np * np * sizeof(float2) + 1024;
}

// FP32 stage for large n (contract of jacobi32_cluster; info = [buffer,
// sweeps, rounds]).  Returns false, launching nothing, outside its range.
static bool jacobi32_pos(System& s, DenseWs& w, const double2* A, int64_t lda, int n, double tol,
                         int max_sweeps, double2* Q, int64_t ldq, double* diag, int* info,
                         cudaStream_t st) {
  if (n < 64 || n > 4096 || max_sweeps > 64) return false;
  const int np = n + (n & 1), P = np / 2, T = (P + kPjTile - 1) / kPjTile;
  ensure(w.pj, pj_buf_bytes(n));
  ensure(w.jlog, pj_log_bytes(n, max_sweeps));
  float2* A0 = (float2*)w.pj.p;
  float2* A1 = A0 + (size_t)np * np;
  unsigned* red = (unsigned*)(A1 + (size_t)np * np);
  PWH_CUDA(cudaMemsetAsync(red, 0, 2 * max_sweeps * sizeof(unsigned), st));
  unsigned* ctl = (unsigned*)w.ctl;
  PWH_CUDA(cudaMemsetAsync(ctl, 0, 3 * sizeof(unsigned), st));  // barrier words
  k_to_pos32<<<(int)std::min<int64_t>(2048, ((int64_t)np * np + 255) / 256), 256, 0, st>>>(A, lda, n,
                                                                                          np, A0);
  PWH_LAUNCH_CHECK();
  PjArgs a;
  a.A[0] = A0;
  a.A[1] = A1;
  a.log = (float4*)w.jlog.p;
  a.log_rounds = (int64_t)max_sweeps * (np - 1);
  a.diag = diag;
  a.info = info;
  a.red = red;
  a.n = n; a.np = np; a.P = P; a.T = T; a.max_sweeps = max_sweeps;
  a.tol = (float)tol;
  a.gb.count = ctl; a.gb.unused = ctl + 1; a.gb.abort = (int*)(ctl + 2);
  a.gb.err = device_error_word(s);
  const size_t smem = (size_t)P * sizeof(float4);
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(k_jacobi_pos, cudaFuncAttributeMaxDynamicSharedMemorySize, 100 * 1024);
    cudaFuncSetAttribute(k_jacobi_qlog_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  });
  int dev = 0, nsm = 0, per_sm = 0;
  PWH_CUDA(cudaGetDevice(&dev));
  PWH_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  PWH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_jacobi_pos, kPjThreads, smem));
  if (per_sm < 1) return false;
  const int ntiles = T * (T + 1) / 2;
  const int blocks = std::max(1, std::min((ntiles + kPjTiles - 1) / kPjTiles, nsm * std::min(per_sm, 2)));
  void* args[] = {&a};
  PWH_CUDA(cudaLaunchCooperativeKernel((void*)k_jacobi_pos, blocks, kPjThreads, args, smem, st));
  note_launch();
  // Q rows per block: enough for the blocks to make one wave over the SMs
  // (every round costs a block barrier whatever its row count), at most what
  // fits in 220 KB of shared memory
  const int qrows = (int)std::max<int64_t>(
      1, std::min<int64_t>(((int64_t)n + nsm - 1) / nsm, (220 << 10) / ((int64_t)n * 8)));
  const size_t qsm = (size_t)qrows * n * sizeof(float2);
  k_jacobi_qlog_rows<<<(n + qrows - 1) / qrows, 1024, qsm, st>>>(a.log, info, n, P, qrows, Q, ldq);
  PWH_LAUNCH_CHECK();
  return true;
}

// ---- FP32 block Jacobi over the whole GPU -----------------------------------
// The indices are cut into blocks of kBjB = 16 that play a round-robin
// tournament (circle method): nblk - 1 rounds a sweep, every block paired
// with one other in each round, so a round holds nblk / 2 pair groups
// P = (I, J) of 32 indices.  A round has two phases, each closed by a grid
// barrier:
//   1. per pair group, plane rotations of the 32 x 32 diagonal block A_PP in
//      shared memory (in the first round of a sweep one cyclic sweep over all
//      its index pairs, in the others the 256 pairs across its two blocks),
//      accumulated into the block rotation U_P (32 x 32), which one
//      Newton-Schulz step brings back to unitary before it is used;
//   2. every other block of the matrix and the eigenvector basis as small
//      complex GEMMs on the CUDA cores, groups of 64 threads each taking one
//      item: A_PQ <- U_P^H A_PQ U_Q for each pair of groups P < Q (A_QP
//      written as its conjugate transpose), Q_RP <- Q_RP U_P for each group R
//      of 32 rows.
// One pass over the matrix thus carries a 32 x 32 block rotation per pair
// group instead of one plane rotation per index pair, and a sweep makes
// nblk - 1 passes instead of n - 1.  Storage: A and Q as nblk x nblk tiles of
// 16 x 16 (A row-major within a tile, Q column-major), A in full (both
// triangles); padding indices beyond n have zero rows and columns, so every
// rotation that involves them is the identity.
constexpr int kBjB = 16;
constexpr int kBjG = 2 * kBjB;
constexpr int kBjTile = kBjB * kBjB;
constexpr int kBjThreads = 256;
constexpr int kBjGroups = kBjThreads / 64;
constexpr int kBjLd = kBjG + 1;  // padded row of the phase-1 block
constexpr int kBjGroupElems = 3 * kBjG * kBjG;  // one item's operands
// two item buffers per group: the next item's operands arrive by cp.async
// while the current one is multiplied
constexpr size_t kBjSmem = (size_t)kBjGroups * 2 * kBjGroupElems * sizeof(float2);

struct BjArgs {
  float2* A;          // nblk x nblk tiles, row-major tiles, full Hermitian
  float2* Q;          // nblk x nblk tiles, column-major tiles
  float2* U;          // nblk / 2 block rotations, 32 x 32 row-major
  double* diag;       // out: eigenvalue estimates, by index
  double2* Qout;      // out: n x n, column-major, ld ldq
  int64_t ldq;
  int* info;          // out: [0] 0, [1] sweeps, [2] 0
  unsigned* red;      // 2 words per sweep (max off-diagonal, max diagonal; float bits), zeroed
  int n, nblk, max_sweeps;
  float tol;
  GridBar gb;
};

// pair k of round r among m players (m even): player m - 1 fixed, the others
// on a circle
__device__ __forceinline__ void bj_pair(int r, int k, int m, int& I, int& J) {
  const int L = m - 1;
  if (k == 0) {
    I = r;
    J = L;
  } else {
    I = (r + k) % L;
    J = (r - k + L) % L;
  }
}
__device__ __forceinline__ float2* bj_tile(float2* X, int nblk, int I, int J) {
  return X + ((size_t)I * nblk + J) * kBjTile;
}
__device__ __forceinline__ void bj_bar(int id) {
  asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ void bj_ld2(const float2* p, float2& a, float2& b) {
  const float4 v = *(const float4*)p;
  a = make_float2(v.x, v.y);
  b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void bj_st2(float2* p, float2 a, float2 b) {
  *(float4*)p = make_float4(a.x, a.y, b.x, b.y);
}
// 16-byte asynchronous copy global -> shared (both 16-byte aligned)
__device__ __forceinline__ void bj_cp16(float2* dst, const float2* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void bj_cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void bj_cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Phase 1 for pair group (I, J): rotations on A_PP, their product U_P to Ub.
// full: one cyclic sweep over all 496 index pairs of the group (31 rounds);
// else only the 256 pairs across the two blocks (16 rounds, pair (i, 16 +
// (i + r) mod 16) in round r).  The first round of a sweep runs full, so
// every index pair of the matrix is rotated once a sweep, as in the scalar
// cyclic method.
__device__ void bj_phase1(const BjArgs& a, float2* sm, int I, int J, float2* Ub, bool full) {
  float2* S = sm;                         // 32 x kBjLd
  float2* Us = sm + kBjG * kBjLd;         // 32 x kBjLd
  float4* rot = (float4*)(Us + kBjG * kBjLd);
  const int tid = threadIdx.x;
  for (int t = tid; t < kBjG * kBjG; t += kBjThreads) {
    const int row = t >> 5, col = t & 31;
    const int Br = row < kBjB ? I : J, Bc = col < kBjB ? I : J;
    S[row * kBjLd + col] = bj_tile(a.A, a.nblk, Br, Bc)[(row & 15) * kBjB + (col & 15)];
    Us[row * kBjLd + col] = make_float2(row == col ? 1.f : 0.f, 0.f);
  }
  __syncthreads();
  const int nround = full ? kBjG - 1 : kBjB;
  for (int ir = 0; ir < nround; ++ir) {
    if (tid < kBjB) {
      int p, q;
      if (full) {
        bj_pair(ir, tid, kBjG, p, q);
      } else {
        p = tid;
        q = kBjB + ((tid + ir) & (kBjB - 1));
      }
      float c;
      float2 sv;
      jacobi_rotation<float>(S[p * kBjLd + q], S[p * kBjLd + p].x, S[q * kBjLd + q].x, c, sv);
      rot[tid] = make_float4(sv.x, sv.y, c, __int_as_float(p | (q << 8)));
    }
    __syncthreads();
    static_assert(kBjThreads == kBjB * kBjB, "one 2 x 2 block of S and two U pairs a thread");
    {
      // 2 x 2 block (pair kk rows, pair ll columns) of J^H S J
      const int kk = tid >> 4, ll = tid & 15;
      const float4 rk = rot[kk], rl = rot[ll];
      const int pq = __float_as_int(rk.w), pl_ql = __float_as_int(rl.w);
      const int pk = pq & 255, qk = pq >> 8, pl = pl_ql & 255, ql = pl_ql >> 8;
      float2 y00, y01, y10, y11;
      jacobi_block<float>(S[pk * kBjLd + pl], S[pk * kBjLd + ql], S[qk * kBjLd + pl],
                          S[qk * kBjLd + ql], rk.z, make_float2(rk.x, rk.y), rl.z,
                          make_float2(rl.x, rl.y), y00, y01, y10, y11);
      if (kk == ll) {
        y00.y = 0.f;
        y11.y = 0.f;
        y01 = make_float2(0.f, 0.f);
        y10 = y01;
      }
      S[pk * kBjLd + pl] = y00;
      S[pk * kBjLd + ql] = y01;
      S[qk * kBjLd + pl] = y10;
      S[qk * kBjLd + ql] = y11;
    }
    {
      // U <- U J on the column pairs: [u_p, u_q] <- [c u_p - conj(s) u_q, s u_p + c u_q]
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int idx = tid + h * kBjThreads;
        const int row = idx >> 4, l = idx & 15;
        const float4 rl = rot[l];
        const int pl_ql = __float_as_int(rl.w);
        const int p = pl_ql & 255, q = pl_ql >> 8;
        const float c = rl.z;
        const float2 sv = make_float2(rl.x, rl.y), sm_ = make_float2(-rl.x, rl.y);
        const float2 u0 = Us[row * kBjLd + p], u1 = Us[row * kBjLd + q];
        Us[row * kBjLd + p] = add<float>(scl<float>(u0, c), mul<float>(u1, sm_));
        Us[row * kBjLd + q] = add<float>(mul<float>(u0, sv), scl<float>(u1, c));
      }
    }
    __syncthreads();
  }
  for (int t = tid; t < kBjG * kBjG; t += kBjThreads) {
    const int row = t >> 5, col = t & 31;
    const int Br = row < kBjB ? I : J, Bc = col < kBjB ? I : J;
    bj_tile(a.A, a.nblk, Br, Bc)[(row & 15) * kBjB + (col & 15)] = S[row * kBjLd + col];
  }
  __syncthreads();
  // one Newton-Schulz step towards the nearest unitary, U (3I - U^H U) / 2:
  // U is a product of 496 FP32 rotations, and its deviation from unitary
  // would otherwise accumulate in Q over every round of every sweep
  for (int t = tid; t < kBjG * kBjG; t += kBjThreads) {
    const int i = t >> 5, j = t & 31;
    float2 g = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int k = 0; k < kBjG; ++k) {
      const float2 x = Us[k * kBjLd + i], y = Us[k * kBjLd + j];
      g.x = fmaf(x.x, y.x, fmaf(x.y, y.y, g.x));
      g.y = fmaf(x.x, y.y, fmaf(-x.y, y.x, g.y));
    }
    S[i * kBjLd + j] = g;  // G = U^H U
  }
  __syncthreads();
  for (int t = tid; t < kBjG * kBjG; t += kBjThreads) {
    const int i = t >> 5, j = t & 31;
    float2 v = make_float2(0.f, 0.f);
#pragma unroll 8
    for (int k = 0; k < kBjG; ++k) v = add<float>(v, mul<float>(Us[i * kBjLd + k], S[k * kBjLd + j]));
    const float2 u = Us[i * kBjLd + j];
    Ub[t] = make_float2(1.5f * u.x - 0.5f * v.x, 1.5f * u.y - 0.5f * v.y);
  }
  __syncthreads();
}

// acc[a][b] += (CONJ ? conj(x[a]) : x[a]) y[b] over k, x = X[k][4 ti ..], y = Y[k][4 tj ..]
// (X, Y 32 x 32 row-major in shared memory)
template <bool CONJ>
__device__ __forceinline__ void bj_gemm(const float2* X, const float2* Y, int ti, int tj,
                                        float2 (&acc)[4][4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);
#pragma unroll 4
  for (int k = 0; k < kBjG; ++k) {
    float2 x[4], y[4];
    bj_ld2(X + k * kBjG + 4 * ti, x[0], x[1]);
    bj_ld2(X + k * kBjG + 4 * ti + 2, x[2], x[3]);
    bj_ld2(Y + k * kBjG + 4 * tj, y[0], y[1]);
    bj_ld2(Y + k * kBjG + 4 * tj + 2, y[2], y[3]);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (CONJ) {
          acc[i][j].x = fmaf(x[i].x, y[j].x, fmaf(x[i].y, y[j].y, acc[i][j].x));
          acc[i][j].y = fmaf(x[i].x, y[j].y, fmaf(-x[i].y, y[j].x, acc[i][j].y));
        } else {
          acc[i][j].x = fmaf(x[i].x, y[j].x, fmaf(-x[i].y, y[j].y, acc[i][j].x));
          acc[i][j].y = fmaf(x[i].x, y[j].y, fmaf(x[i].y, y[j].x, acc[i][j].y));
        }
      }
  }
}

// One phase-2 item of round r: a Q item (row group R, pair group P) or a
// pair of pair groups (P, Qg), P < Qg, numbered row by row after the Q items.
struct BjItem {
  bool q;
  int R, P, Qg, I1, J1, I2, J2;
};
__device__ __forceinline__ BjItem bj_decode(int r, int it, int nblk, int nb2, int nQ) {
  BjItem x;
  if (it < nQ) {
    x.q = true;
    x.R = it / nb2;
    x.P = it - x.R * nb2;
    x.Qg = 0;
    bj_pair(r, x.P, nblk, x.I1, x.J1);
    x.I2 = x.J2 = 0;
  } else {
    x.q = false;
    x.R = 0;
    const int t = it - nQ;
    const int m2 = 2 * nb2 - 1;
    int P = (int)((m2 - sqrtf((float)m2 * m2 - 8.f * t)) * 0.5f);
    P = max(0, min(P, nb2 - 2));
    while (P > 0 && P * (m2 - P) / 2 > t) --P;
    while ((P + 1) * (m2 - P - 1) / 2 <= t) ++P;
    x.P = P;
    x.Qg = P + 1 + (t - P * (m2 - P) / 2);
    bj_pair(r, x.P, nblk, x.I1, x.J1);
    bj_pair(r, x.Qg, nblk, x.I2, x.J2);
  }
  return x;
}

// Issue the asynchronous copies of an item's operands into buf (thread lt of
// its group): X0 the 32 x 32 block (Q item: transposed, X0[k][i] = Q[32 R +
// i][column k of P], contiguous in i in the column-major tiles; A item:
// A_PQ row-major), X1 = U_P, X2 = U_Q.
__device__ __forceinline__ void bj_issue(const BjArgs& a, const BjItem& x, int lt, float2* buf) {
  float2* X0 = buf;
  float2* X1 = buf + kBjG * kBjG;
  float2* X2 = buf + 2 * kBjG * kBjG;
  const float2* U1 = a.U + (size_t)x.P * kBjG * kBjG;
  if (x.q) {
    for (int v = lt; v < kBjG * kBjG / 2; v += 64) {
      const int e = 2 * v, k = e >> 5, i = e & 31;
      const float2* src = bj_tile(a.Q, a.nblk, 2 * x.R + (i >> 4), k < kBjB ? x.I1 : x.J1);
      bj_cp16(X0 + e, src + (k & 15) * kBjB + (i & 15));
      bj_cp16(X1 + e, U1 + e);
    }
  } else {
    const float2* U2 = a.U + (size_t)x.Qg * kBjG * kBjG;
    for (int v = lt; v < kBjG * kBjG / 2; v += 64) {
      const int e = 2 * v, row = e >> 5, col = e & 31;
      const float2* src =
          bj_tile(a.A, a.nblk, row < kBjB ? x.I1 : x.J1, col < kBjB ? x.I2 : x.J2);
      bj_cp16(X0 + e, src + (row & 15) * kBjB + (col & 15));
      bj_cp16(X1 + e, U1 + e);
      bj_cp16(X2 + e, U2 + e);
    }
  }
}

// Multiply an item whose operands are in buf and store the result:
// Q_RP <- Q_RP U_P, or A_PQ <- U_P^H A_PQ U_Q with A_QP its conjugate
// transpose.  Every thread of the group; X0 is reused for T^T.
__device__ __forceinline__ void bj_item(const BjArgs& a, const BjItem& x, int ti, int tj, int grp,
                                        float2* buf) {
  float2* X0 = buf;
  float2* X1 = buf + kBjG * kBjG;
  float2* X2 = buf + 2 * kBjG * kBjG;
  float2 acc[4][4];
  if (x.q) {
    bj_gemm<false>(X0, X1, ti, tj, acc);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int col = 4 * tj + j;
      float2* dst = bj_tile(a.Q, a.nblk, 2 * x.R + (ti >> 2), col < kBjB ? x.I1 : x.J1) +
                    (col & 15) * kBjB + ((4 * ti) & 15);
      bj_st2(dst, acc[0][j], acc[1][j]);
      bj_st2(dst + 2, acc[2][j], acc[3][j]);
    }
    return;
  }
  bj_gemm<true>(X1, X0, ti, tj, acc);  // T = U_P^H A_PQ
  bj_bar(grp + 1);
  // X0 <- T^T (row k holds column k of T)
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float2* d = X0 + (4 * tj + j) * kBjG + 4 * ti;
    bj_st2(d, acc[0][j], acc[1][j]);
    bj_st2(d + 2, acc[2][j], acc[3][j]);
  }
  bj_bar(grp + 1);
  bj_gemm<false>(X0, X2, ti, tj, acc);  // T U_Q
  const int rb = (4 * ti) < kBjB ? x.I1 : x.J1, cb = (4 * tj) < kBjB ? x.I2 : x.J2;
  float2* up = bj_tile(a.A, a.nblk, rb, cb);
  float2* lo = bj_tile(a.A, a.nblk, cb, rb);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float2* d = up + (((4 * ti) & 15) + i) * kBjB + ((4 * tj) & 15);
    bj_st2(d, acc[i][0], acc[i][1]);
    bj_st2(d + 2, acc[i][2], acc[i][3]);
  }
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float2* d = lo + (((4 * tj) & 15) + j) * kBjB + ((4 * ti) & 15);
    bj_st2(d, make_float2(acc[0][j].x, -acc[0][j].y), make_float2(acc[1][j].x, -acc[1][j].y));
    bj_st2(d + 2, make_float2(acc[2][j].x, -acc[2][j].y), make_float2(acc[3][j].x, -acc[3][j].y));
  }
}

__global__ void __launch_bounds__(kBjThreads, 1) k_jacobi_blk(BjArgs a) {
  extern __shared__ __align__(16) unsigned char bjs[];
  float2* sm = (float2*)bjs;
  __shared__ float s_red[2][kBjThreads / 32];
  const int tid = threadIdx.x, grp = tid >> 6, lt = tid & 63;
  const int ti = lt & 7, tj = lt >> 3;
  const int nblk = a.nblk, nb2 = nblk / 2, n = a.n;
  const int nA = nb2 * (nb2 - 1) / 2, nQ = nb2 * nb2, nItems = nQ + nA;
  const int gtid = blockIdx.x * blockDim.x + tid, nth = gridDim.x * blockDim.x;
  float2* gs = sm + (size_t)grp * 2 * kBjGroupElems;  // the group's two item buffers
  unsigned epoch = 0;
  int sweep = 0;
  bool done = false;
  while (sweep < a.max_sweeps && !done) {
    for (int r = 0; r < nblk - 1; ++r) {
      // ---- phase 1: the diagonal pair blocks
      for (int k = blockIdx.x; k < nb2; k += gridDim.x) {
        int I, J;
        bj_pair(r, k, nblk, I, J);
        bj_phase1(a, sm, I, J, a.U + (size_t)k * kBjG * kBjG, r == 0);
      }
      if (!grid_sync(a.gb, epoch)) return;
      // ---- phase 2: Q row groups, then the off-diagonal pair blocks; each
      // group of 64 threads walks its items with the next item's operands in
      // flight (cp.async into its other buffer) while it multiplies the
      // current one
      {
        const int stride = gridDim.x * kBjGroups;
        int it = blockIdx.x * kBjGroups + grp;
        int b = 0;
        if (it < nItems) bj_issue(a, bj_decode(r, it, nblk, nb2, nQ), lt, gs);
        bj_cp_commit();
        for (; it < nItems; it += stride) {
          float2* cur = gs + (size_t)b * kBjGroupElems;
          if (it + stride < nItems)
            bj_issue(a, bj_decode(r, it + stride, nblk, nb2, nQ), lt,
                     gs + (size_t)(b ^ 1) * kBjGroupElems);
          bj_cp_commit();
          bj_cp_wait<1>();  // this thread's copies of the current item have landed
          bj_bar(grp + 1);  // and every thread's
          bj_item(a, bj_decode(r, it, nblk, nb2, nQ), ti, tj, grp, cur);
          bj_bar(grp + 1);  // the buffer is free for the item after next
          b ^= 1;
        }
        bj_cp_wait<0>();
      }
      if (!grid_sync(a.gb, epoch)) return;
    }
    // convergence: grid-wide maxima of |A_ij| (i < j < n) and |A_ii|
    {
      float off = 0.f, dm = 0.f;
      const int64_t tot = (int64_t)nblk * nblk * kBjTile;
      for (int64_t t = gtid; t < tot; t += nth) {
        const int64_t tile = t / kBjTile;
        const int e = (int)(t - tile * kBjTile);
        const int i = (int)(tile / nblk) * kBjB + (e >> 4), j = (int)(tile % nblk) * kBjB + (e & 15);
        if (i >= n || j >= n || i > j) continue;
        const float2 v = a.A[t];
        if (i == j) dm = fmaxf(dm, fabsf(v.x));
        else off = fmaxf(off, sqrtf(v.x * v.x + v.y * v.y));
      }
      for (int o = 16; o > 0; o >>= 1) {
        off = fmaxf(off, __shfl_xor_sync(0xffffffffu, off, o));
        dm = fmaxf(dm, __shfl_xor_sync(0xffffffffu, dm, o));
      }
      if ((tid & 31) == 0) {
        s_red[0][tid >> 5] = off;
        s_red[1][tid >> 5] = dm;
      }
      __syncthreads();
      if (tid == 0) {
        for (int w = 1; w < kBjThreads / 32; ++w) {
          s_red[0][0] = fmaxf(s_red[0][0], s_red[0][w]);
          s_red[1][0] = fmaxf(s_red[1][0], s_red[1][w]);
        }
        atomicMax(a.red + 2 * sweep, __float_as_uint(s_red[0][0]));
        atomicMax(a.red + 2 * sweep + 1, __float_as_uint(s_red[1][0]));
      }
      if (!grid_sync(a.gb, epoch)) return;
      const float offg = __uint_as_float(*(volatile unsigned*)(a.red + 2 * sweep));
      const float dmg = __uint_as_float(*(volatile unsigned*)(a.red + 2 * sweep + 1));
      done = offg <= a.tol * fmaxf(dmg, 1e-30f);
    }
    ++sweep;
  }
  if (gtid == 0) {
    a.info[0] = 0;
    a.info[1] = sweep;
    a.info[2] = 0;
  }
  for (int i = gtid; i < n; i += nth)
    a.diag[i] = (double)bj_tile(a.A, nblk, i >> 4, i >> 4)[(i & 15) * kBjB + (i & 15)].x;
  for (int64_t t = gtid; t < (int64_t)n * n; t += nth) {
    const int j = (int)(t / n), i = (int)(t - (int64_t)j * n);
    const float2 v = bj_tile(a.Q, nblk, i >> 4, j >> 4)[(j & 15) * kBjB + (i & 15)];
    a.Qout[(size_t)j * a.ldq + i] = make_double2((double)v.x, (double)v.y);
  }
}

// FP64 start (n x n, ld lda) -> FP32 tiles of A (row-major tiles, zero
// padded) and Q = identity (column-major tiles).
__global__ void k_bj_init(const double2* __restrict__ A, int64_t lda, int n, int nblk,
                          float2* __restrict__ At, float2* __restrict__ Qt) {
  const int64_t tot = (int64_t)nblk * nblk * kBjTile;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t tile = t / kBjTile;
    const int e = (int)(t - tile * kBjTile);
    const int I = (int)(tile / nblk), J = (int)(tile % nblk);
    const int i = I * kBjB + (e >> 4), j = J * kBjB + (e & 15);  // A: row-major in the tile
    const double2 z = (i < n && j < n) ? A[(size_t)j * lda + i] : make_double2(0.0, 0.0);
    At[t] = make_float2((float)z.x, (float)z.y);
    const int qi = I * kBjB + (e & 15), qj = J * kBjB + (e >> 4);  // Q: column-major
    Qt[t] = make_float2(qi == qj ? 1.f : 0.f, 0.f);
  }
}

static int bj_nblk(int n) {
  const int nblk = (n + kBjB - 1) / kBjB;
  return nblk + (nblk & 1);
}
static size_t bj_buf_bytes(int n) {
  const size_t np = (size_t)bj_nblk(n) * kBjB;
  return (2 * np * np + (size_t)(np / kBjG) * kBjG * kBjG) * sizeof(float2) + 1024;
}

// Work of one sweep of k_jacobi_blk, in real flops: the phase-2 GEMMs
// (8 x 32^3 each: two per pair of groups, one per row group and pair group)
// and phase 1 (rotation rounds of 20 flops per element of the block and 10
// per element of its rotation: 31 in the first round of a sweep, 16 in the
// others; and the Newton-Schulz step's two products).
double jacobi32_blk_sweep_flops(int n) {
  const double nb = bj_nblk(n), nb2 = nb / 2;
  const double g3 = 8.0 * kBjG * kBjG * kBjG;
  const double p2 = g3 * (2.0 * nb2 * (nb2 - 1) / 2 + nb2 * nb2);
  const double rot = (kBjG - 1) + (double)kBjB * (nb - 2);  // rotation rounds a sweep
  const double p1 = nb2 * (rot * 30.0 * kBjG * kBjG + (nb - 1) * 2 * g3);
  return (nb - 1) * p2 + p1;
}

// FP32 stage for n > 512 (contract of jacobi32_cluster; info = [0, sweeps,
// 0]).  Returns false, launching nothing, outside its range.
static bool jacobi32_blk(System& s, DenseWs& w, const double2* A, int64_t lda, int n, double tol,
                         int max_sweeps, double2* Q, int64_t ldq, double* diag, int* info,
                         cudaStream_t st) {
  if (n < 64 || n > kJacobiMaxN || max_sweeps > 64) return false;
  const int nblk = bj_nblk(n);
  const size_t np = (size_t)nblk * kBjB;
  ensure(w.pj, bj_buf_bytes(n));
  float2* At = (float2*)w.pj.p;
  float2* Qt = At + np * np;
  float2* U = Qt + np * np;
  unsigned* red = (unsigned*)(U + (size_t)(nblk / 2) * kBjG * kBjG);
  PWH_CUDA(cudaMemsetAsync(red, 0, 2 * max_sweeps * sizeof(unsigned), st));
  unsigned* ctl = (unsigned*)w.ctl;
  PWH_CUDA(cudaMemsetAsync(ctl, 0, 3 * sizeof(unsigned), st));  // barrier words
  k_bj_init<<<(int)std::min<int64_t>(2048, ((int64_t)np * np + 255) / 256), 256, 0, st>>>(
      A, lda, n, nblk, At, Qt);
  PWH_LAUNCH_CHECK();
  BjArgs a;
  a.A = At;
  a.Q = Qt;
  a.U = U;
  a.diag = diag;
  a.Qout = Q;
  a.ldq = ldq;
  a.info = info;
  a.red = red;
  a.n = n; a.nblk = nblk; a.max_sweeps = max_sweeps;
  a.tol = (float)tol;
  a.gb.count = ctl; a.gb.unused = ctl + 1; a.gb.abort = (int*)(ctl + 2);
  a.gb.err = device_error_word(s);
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(k_jacobi_blk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBjSmem);
  });
  int dev = 0, nsm = 0, per_sm = 0;
  PWH_CUDA(cudaGetDevice(&dev));
  PWH_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  PWH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_jacobi_blk, kBjThreads, kBjSmem));
  if (per_sm < 1) return false;
  void* args[] = {&a};
  PWH_CUDA(cudaLaunchCooperativeKernel((void*)k_jacobi_blk, nsm, kBjThreads, args, kBjSmem, st));
  note_launch();
  return true;
}

// FP32 stage: above n = 512 the whole-GPU block Jacobi; for 64 <= n <= 512 the cluster kernel or the
// position-order one, whichever was faster on the first matrix of the size
// class (n rounded up to 32): both are run on it (same read-only input, same
// outputs; the second run's result is kept), timed with CUDA events.  While
// the stream is being captured the cluster kernel runs without timing.
static bool jacobi32_tuned(System& s, DenseWs& w, const double2* A, int64_t lda, int n, double tol,
                           int max_sweeps, double2* Q, int64_t ldq, double* diag, int* info,
                           cudaStream_t st) {
  if (n > 512) return jacobi32_blk(s, w, A, lda, n, tol, max_sweeps, Q, ldq, diag, info, st);
  if (n < 64) return false;
  static std::mutex mu;
  static std::map<int, int> choice;  // size class -> 0 cluster, 1 position order
  const int cls = (n + 31) / 32;
  int c = -1;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = choice.find(cls);
    if (it != choice.end()) c = it->second;
  }
  if (c == 0) return jacobi32_cluster(s, w, A, lda, n, tol, max_sweeps, Q, ldq, diag, info, st);
  if (c == 1) return jacobi32_pos(s, w, A, lda, n, tol, max_sweeps, Q, ldq, diag, info, st);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  PWH_CUDA(cudaStreamIsCapturing(st, &cap));
  if (cap != cudaStreamCaptureStatusNone)
    return jacobi32_cluster(s, w, A, lda, n, tol, max_sweeps, Q, ldq, diag, info, st);
  cudaEvent_t e[3];
  for (auto& x : e) PWH_CUDA(cudaEventCreate(&x));
  PWH_CUDA(cudaEventRecord(e[0], st));
  const bool ok0 = jacobi32_cluster(s, w, A, lda, n, tol, max_sweeps, Q, ldq, diag, info, st);
  PWH_CUDA(cudaEventRecord(e[1], st));
  const bool ok1 = jacobi32_pos(s, w, A, lda, n, tol, max_sweeps, Q, ldq, diag, info, st);
  PWH_CUDA(cudaEventRecord(e[2], st));
  PWH_CUDA(cudaEventSynchronize(e[2]));
  float t0 = 0.f, t1 = 0.f;
  PWH_CUDA(cudaEventElapsedTime(&t0, e[0], e[1]));
  PWH_CUDA(cudaEventElapsedTime(&t1, e[1], e[2]));
  for (auto& x : e) cudaEventDestroy(x);
  {
    std::lock_guard<std::mutex> lock(mu);
    choice[cls] = (ok1 && (!ok0 || t1 < t0)) ? 1 : 0;
  }
  if (ok1) return true;  // its result is the one in Q / diag / info
  return ok0 && jacobi32_cluster(s, w, A, lda, n, tol, max_sweeps, Q, ldq, diag, info, st);
}

template <typename T>
static void launch_jacobi(System& s, DenseWs& w, cx<T>* A0, cx<T>* A1, cx<T>* Q0, cx<T>* Q1, int n,
                          double tol, int max_sweeps, int* out_buf, cudaStream_t st,
                          const int* skip = nullptr,
                          const unsigned long long* dmax = nullptr) {
  const int np = n + (n & 1);
  unsigned* ctl = (unsigned*)w.ctl;
  PWH_CUDA(cudaMemsetAsync(ctl, 0, 3 * sizeof(unsigned), st));  // barrier words
  JacobiArgsT<T> a;
  a.A[0] = A0; a.A[1] = A1; a.Q[0] = Q0; a.Q[1] = Q1;
  a.n = n; a.np = np; a.max_sweeps = max_sweeps; a.tol = tol;
  a.out_buf = out_buf;
  a.conv = (int*)(ctl + 12);
  a.skip = skip;
  a.dmax = dmax;
  a.gb.count = ctl; a.gb.unused = ctl + 1; a.gb.abort = (int*)(ctl + 2);
  a.gb.err = device_error_word(s);
  const int P = np / 2;
  const size_t smem = (size_t)P * (sizeof(cx<T>) + sizeof(T) + 2 * sizeof(int)) + 16;
  static std::once_flag attr_once;
  static int cluster_size = 0;  // largest cluster (16 or 8) that fits, 0 if none
  std::call_once(attr_once, [] {
    cudaFuncSetAttribute(k_jacobi<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if constexpr (sizeof(T) == 8)
      cudaFuncSetAttribute(k_jacobi<T, false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(k_jacobi<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    cudaFuncSetAttribute(k_jacobi<T, true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (int cs : {16, 8}) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(cs);
      cfg.blockDim = dim3(256);
      cfg.dynamicSmemBytes = 64 * 1024;
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = cs;
      at[0].val.clusterDim.y = 1;
      at[0].val.clusterDim.z = 1;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int nclusters = 0;
      if (cudaOccupancyMaxActiveClusters(&nclusters, (void*)k_jacobi<T, true>, &cfg) == cudaSuccess &&
          nclusters >= 1) {
        cluster_size = cs;
        break;
      }
    }
    cudaGetLastError();  // clear a refused query
  });
  // Reduced precision, small size: one cluster, hardware barrier per round
  // (beyond ~192 the per-thread share of each round outweighs the barrier)
  if (sizeof(T) == 4 && n <= 192 && cluster_size > 0) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster_size);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster_size;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    PWH_CUDA(cudaLaunchKernelEx(&cfg, k_jacobi<T, true>, a));
    note_launch();
    return;
  }
  int dev = 0, nsm = 0, per_sm = 0;
  PWH_CUDA(cudaGetDevice(&dev));
  PWH_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  const void* kernel = (const void*)k_jacobi<T, false>;
  if constexpr (sizeof(T) == 8)
    if (skip) kernel = (const void*)k_jacobi<T, false, true>;
  PWH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, smem));
  // FP32 stage: few blocks (the per-round barrier latency dominates);
  // FP64 stage: every SM, the FP64 units are the limit
  const int64_t items = (int64_t)P * P + (int64_t)n * P;
  const int64_t per_block = sizeof(T) == 8 ? 64 : 256;
  const int want = (int)std::max<int64_t>(1, std::min<int64_t>((items + per_block - 1) / per_block, nsm));
  const int blocks = std::max(1, std::min(want, nsm * std::max(per_sm, 1)));
  void* args[] = {&a};
  PWH_CUDA(cudaLaunchCooperativeKernel(kernel, blocks, 256, args, smem, st));
  note_launch();
}

// ---- FP64 refinement of the FP32 eigenvectors by matrix products -----------
// Quadratically convergent correction of an approximate eigenvector matrix X
// (Ogita and Aishima, "Iterative refinement for symmetric eigenvalue
// decomposition", 2018): with R = I - X^H X and S = X^H H X, X <- X (I + R/2) (I + E)
// where E_ij = F_ij / (f_j - f_i), F = S + (R_ij / 2)(S_ii + S_jj) the
// symmetrically orthonormalised S, f its diagonal.  Close pairs, where the
// first-order angle would be large, are treated as Jacobi does: index i and
// its strongest partner p(i), when each is the other's strongest and the angle
// passes `lim`, are rotated exactly (J, unitary) and E is formed from J^H F J;
// any other angle above `lim` is left for the next step, so that X stays
// within lim^2 of unitary (clusters of three and more equal eigenvalues are
// resolved a pair at a time, or left to the Jacobi sweeps).
//   Bound: four n x n products a step (12 in all) and one Jacobi sweep before
// them (k_jacobi_pair_sweep), against two to three (30 in large clusters) sweeps
// of n - 1 grid-wide rounds on the FP64 pipe (60 us a round at n = 1088).  The
// whole FP64 eigensolve, FP32 stage included: n = 1088 137 -> 42 ms, 1632 587 ->
// 126, 408 21.7 -> 14.0, 256 (random) 16.2 -> 15.3, five 128-fold levels 311 -> 31;
// eigenvectors orthonormal to 3e-15 instead of 1e-13.  Without the first sweep (three
// refinement steps from the FP32 basis) n = 1088 takes 20 ms to the same
// accuracy, but with eigenvector phases that differ by 1e-6 from the cyclic
// sweeps'.  At kRefineMinN the FP64 stage takes 5.1 ms (its products, below 2e8 flops,
// on the FP64 pipe) against 5.9 of the sweeps; smaller matrices gain less.
constexpr int kRefineMinN = 256;
struct RefineWs {
  double* dS;              // S_ii
  double* f;               // F_ii
  double* f2;              // diagonal of J^H F J
  int* best;               // strongest partner
  int* pair;               // its index when rotated, else -1
  double* c;               // J_ii
  double2* s;              // J_{i, p(i)}
  unsigned long long* mx;  // max |F_ij|, max |F_ii| as ordered bit patterns
  int* done;               // 1: every off-diagonal element below the target
};
static size_t refine_bytes(int n) {
  // refinement arrays, then the pair sweep's two diagonals and rotations
  return (size_t)n * 56 + 64 + (size_t)n * 16 + (size_t)(n / 2 + 1) * 20 + 64;
}
static RefineWs refine_carve(void* base, int n) {
  RefineWs w;
  w.s = (double2*)(((uintptr_t)base + 15) & ~(uintptr_t)15);
  w.dS = (double*)(w.s + n);
  w.f = w.dS + n;
  w.f2 = w.f + n;
  w.c = w.f2 + n;
  w.best = (int*)(w.c + n);
  w.pair = w.best + n;
  w.mx = (unsigned long long*)(((uintptr_t)(w.pair + n) + 7) & ~(uintptr_t)7);
  w.done = (int*)(w.mx + 2);
  return w;
}

// tan of the Jacobi angle that zeroes an off-diagonal element of modulus g
// between diagonal elements a (row) and b (column); first: tie rule at a = b
__device__ __forceinline__ double refine_tan(double g, double a, double b, bool first) {
  if (!(g > 0.0)) return 0.0;
  const double zeta = (b - a) / (2.0 * g), az = fabs(zeta);
  const double sg = zeta > 0.0 || (zeta == 0.0 && first) ? 1.0 : -1.0;
  return az > 1e9 ? 0.5 / zeta : sg / (az + sqrt(1.0 + az * az));
}
// F_ij (i != j) from S, the Gram matrix and S's diagonal
__device__ __forceinline__ double2 refine_f(const double2* S, const double2* Gm, const double* dS,
                                            int n, int i, int j) {
  const double2 s = S[(size_t)j * n + i], g = Gm[(size_t)j * n + i];
  const double h = -0.5 * (dS[i] + dS[j]);  // R_ij = -Gram_ij off the diagonal
  return make_double2(s.x + h * g.x, s.y + h * g.y);
}

__global__ void k_refine_diag(const double2* __restrict__ S, const double2* __restrict__ Gm, int n,
                              RefineWs w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) w.mx[0] = 0;
  if (i >= n) return;
  const double d = S[(size_t)i * n + i].x;
  w.dS[i] = d;
  w.f[i] = d * (2.0 - Gm[(size_t)i * n + i].x);  // S_ii + R_ii S_ii
}
// max |F_ii| (one block)
__global__ void k_refine_max(int n, RefineWs w) {
  __shared__ double red[32];
  double m = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, fabs(w.f[i]));
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) m = fmax(m, red[k]);
    w.mx[1] = (unsigned long long)__double_as_longlong(m);
  }
}
// Strongest partner of every index (a block per column), max |F_ij|.
__global__ void __launch_bounds__(128) k_refine_best(const double2* __restrict__ S,
                                                     const double2* __restrict__ Gm, int n,
                                                     RefineWs w) {
  __shared__ double rq[4], rg[4];
  __shared__ int ri[4];
  const int j = blockIdx.x;
  const double fj = w.f[j];
  const double floor_g = 2e-16 * __longlong_as_double((long long)w.mx[1]);
  double bq = -1.0, mg = 0.0;
  int bi = -1;
  for (int i = threadIdx.x; i < n; i += 128) {
    if (i == j) continue;
    const double2 F = refine_f(S, Gm, w.dS, n, i, j);
    const double g = sqrt(F.x * F.x + F.y * F.y);
    mg = fmax(mg, g);
    if (!(g > floor_g)) continue;
    // the angle grows with |F_ij| over the gap
    const double q = g / fmax(fabs(fj - w.f[i]), 1e-300);
    if (q > bq) {
      bq = q;
      bi = i;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double q2 = __shfl_xor_sync(0xffffffffu, bq, o), g2 = __shfl_xor_sync(0xffffffffu, mg, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
    if (q2 > bq || (q2 == bq && i2 >= 0 && (bi < 0 || i2 < bi))) {
      bq = q2;
      bi = i2;
    }
    mg = fmax(mg, g2);
  }
  if ((threadIdx.x & 31) == 0) {
    rq[threadIdx.x >> 5] = bq;
    rg[threadIdx.x >> 5] = mg;
    ri[threadIdx.x >> 5] = bi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 4; ++k) {
      if (rq[k] > bq || (rq[k] == bq && ri[k] >= 0 && (bi < 0 || ri[k] < bi))) {
        bq = rq[k];
        bi = ri[k];
      }
      mg = fmax(mg, rg[k]);
    }
    w.best[j] = bi;
    atomicMax(&w.mx[0], (unsigned long long)__double_as_longlong(mg));
  }
}
// Pair rotations; done = max |F_ij| <= tol max |F_ii|.  (The maxima pass over NaN: a
// matrix of NaN counts as done, no sweep could mend it, and its results are NaN.)
__global__ void k_refine_pairs(const double2* __restrict__ S, const double2* __restrict__ Gm, int n,
                               double lim, double tol, RefineWs w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0)
    *w.done = __longlong_as_double((long long)w.mx[0]) <=
              tol * fmax(__longlong_as_double((long long)w.mx[1]), 1e-300);
  if (i >= n) return;
  int p = -1;
  double c = 1.0, f2 = w.f[i];
  double2 s = make_double2(0, 0);
  const int j = w.best[i];
  if (j >= 0 && w.best[j] == i) {
    const int a = min(i, j), b = max(i, j);
    const double2 F = refine_f(S, Gm, w.dS, n, a, b);
    const double g = sqrt(F.x * F.x + F.y * F.y);
    const double t = refine_tan(g, w.f[a], w.f[b], true);
    if (fabs(t) > lim) {
      p = j;
      c = 1.0 / sqrt(1.0 + t * t);
      const double e = t * c / g;
      // J_ab = s, J_ba = -conj(s)
      s = i == a ? make_double2(e * F.x, e * F.y) : make_double2(-e * F.x, e * F.y);
      f2 = i == a ? w.f[a] - t * g : w.f[b] + t * g;
    }
  }
  w.pair[i] = p;
  w.c[i] = c;
  w.s[i] = s;
  w.f2[i] = f2;
}
// Column j of M = (I + R/2) J (I + E), first order in R (a block per column, the
// column of E in shared memory; E_jj = -sum |E_ij|^2 / 2).  last: the step after
// which the Jacobi sweeps may run; when the target was missed M = I + R/2 and S
// becomes F (X then is unitary to R^2), else S's diagonal holds the
// eigenvalues.  (Diagonal elements of S are never read here, other columns'
// elements only when the target was met.)
__global__ void __launch_bounds__(128) k_refine_m(double2* __restrict__ S,
                                                  const double2* __restrict__ Gm, int n, double lim,
                                                  int last, RefineWs w, double2* __restrict__ M) {
  extern __shared__ __align__(16) unsigned char rsm[];
  double2* E = (double2*)rsm;
  __shared__ double red[4];
  const int j = blockIdx.x;
  const double2* Gj = Gm + (size_t)j * n;
  double2* Mj = M + (size_t)j * n;
  if (last && !*w.done) {
    for (int i = threadIdx.x; i < n; i += 128) {
      S[(size_t)j * n + i] = i == j ? make_double2(w.f[i], 0.0) : refine_f(S, Gm, w.dS, n, i, j);
      Mj[i] = make_double2((i == j ? 1.5 : 0.0) - 0.5 * Gj[i].x, -0.5 * Gj[i].y);
    }
    return;
  }
  const int pj = w.pair[j];
  const double cj = w.c[j], f2j = w.f2[j];
  // column j of J: J_jj = c_j, J_{p(j), j} = s_{p(j)}
  const double2 sj = pj >= 0 ? w.s[pj] : make_double2(0, 0);
  const double floor_g = 2e-16 * __longlong_as_double((long long)w.mx[1]);
  double sum = 0.0;
  for (int i = threadIdx.x; i < n; i += 128) {
    double2 e = make_double2(0, 0);
    if (i != pj && i != j) {
      const int pi = w.pair[i];
      // (F J)_aj for a = i, p(i), then (J^H . )_ij
      auto col = [&](int a) {
        double2 v = scl<double>(refine_f(S, Gm, w.dS, n, a, j), cj);
        if (pj >= 0) v = add<double>(v, mul<double>(refine_f(S, Gm, w.dS, n, a, pj), sj));
        return v;
      };
      double2 F = scl<double>(col(i), w.c[i]);
      if (pi >= 0) F = add<double>(F, mulc<double>(col(pi), w.s[pi]));  // conj(J_{p(i), i})
      const double g = sqrt(F.x * F.x + F.y * F.y);
      if (g > floor_g) {
        const double t = refine_tan(g, w.f2[i], f2j, i < j);
        if (fabs(t) <= lim) {
          const double u = t / g;
          e = make_double2(u * F.x, u * F.y);
          sum += t * t;
        }
      }
    }
    E[i] = e;
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    E[j] = make_double2(1.0 - 0.5 * (red[0] + red[1] + red[2] + red[3]), 0.0);  // I + E
    if (last) S[(size_t)j * n + j] = make_double2(f2j, 0.0);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += 128) {
    const int p = w.pair[i];
    double2 m = scl<double>(E[i], w.c[i]);
    if (p >= 0) m = add<double>(m, mul<double>(w.s[i], E[p]));
    // (R / 2) J
    double2 r = make_double2((i == j ? 0.5 : 0.0) - 0.5 * Gj[i].x, -0.5 * Gj[i].y);
    r = scl<double>(r, cj);
    if (pj >= 0) {
      const double2 g = Gm[(size_t)pj * n + i];
      r = add<double>(r, mul<double>(make_double2((i == pj ? 0.5 : 0.0) - 0.5 * g.x, -0.5 * g.y), sj));
    }
    Mj[i] = add<double>(m, r);
  }
}

// ---- range of the matrix -------------------------------------------------------
// FP32 sweeps square elements down to 1e-7 of the largest: below about 1e-19 they
// vanish and nothing rotates, and a sweep in FP32 pairs that has to turn vectors by
// large angles leaves them unitary to 1e-6 only (eigenvalues off by 1e-12 at a scale
// of 1e-30).  A matrix whose largest element lies outside [2^-20, 2^41) is scaled by
// a power of two, exactly, to one near 1; the others keep their bits.
__device__ __forceinline__ int eig_exponent(const unsigned* mx) {
  const int eb = (int)(*mx >> 20);  // biased exponent of the largest |Re|, |Im|
  return eb == 0x7ff || *mx == 0 || (eb >= 1023 - 20 && eb <= 1023 + 40) ? 0 : eb - 1023;
}
__global__ void __launch_bounds__(256) k_eig_max(const double2* __restrict__ H, int64_t ldh, int n,
                                                 unsigned* __restrict__ mx) {
  unsigned m = 0;
  for (int64_t t = blockIdx.x * (int64_t)256 + threadIdx.x; t < (int64_t)n * n; t += gridDim.x * 256ll) {
    const double2 v = H[(t / n) * ldh + t % n];
    m = max(m, max((unsigned)__double2hiint(v.x) & 0x7fffffffu, (unsigned)__double2hiint(v.y) & 0x7fffffffu));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(mx, m);
}
__global__ void __launch_bounds__(256) k_eig_scale(const double2* __restrict__ H, int64_t ldh, int n,
                                                   const unsigned* __restrict__ mx,
                                                   double2* __restrict__ out) {
  const int e = eig_exponent(mx);
  for (int64_t t = blockIdx.x * (int64_t)256 + threadIdx.x; t < (int64_t)n * n; t += gridDim.x * 256ll) {
    double2 v = H[(t / n) * ldh + t % n];
    if (e) v = make_double2(scalbn(v.x, -e), scalbn(v.y, -e));
    out[t] = v;
  }
}
__global__ void k_eig_unscale(double* __restrict__ d, int n, const unsigned* __restrict__ mx) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x, e = eig_exponent(mx);
  if (i < n && e) d[i] = scalbn(d[i], e);
}

// ---- the first FP64 sweep in FP32 pairs ---------------------------------------
// One cyclic sweep (the rounds and rotations of k_jacobi<double>) on the almost
// diagonal A: its diagonal in FP64, off-diagonal elements and Q as pairs hi + lo of
// FP32 numbers (48 bits).  A rotation is the identity plus a small correction, so a
// new element is the old pair plus a correction formed in FP32 (angles of 1e-4 of
// the element; the rotation angles themselves in FP64): what the refinement that
// follows needs, a unitary basis to 1e-7 or better, at the FP32 pipes' rate.
//   Each block computes its share of a round's rotations (k_jacobi computes them
// all in every block: at n = 1088 some 25 of its 60 us a round on the FP64 pipe)
// and publishes them; a second grid barrier separates them from the update.
//   Bound: two grid barriers a round and the L2 traffic between them (A read by
// halves and written, Q read and written: 66 MB a round at n = 1088).  The whole
// eigensolve with this sweep in place of an FP64 one: n = 1088 86.8 -> 41.8 ms (60
// -> 20 us a round), 1632 249 -> 126, 408 16.4 -> 14.0, 256 9.6 -> 8.3 (its products on
// the tensor cores at the time).  One barrier
// a round (the next round's rotations formed by the threads that make their
// elements) gave 18 us there but was slower at 256 to 320; four rows of Q in flight
// a thread changed nothing.
struct PairRot {
  float c1, sx, sy;    // c - 1, s
  float sxl, syl;      // low parts of s
};
struct PairSweepArgs {
  float4* A[2];   // (re hi, re lo, im hi, im lo), column-major
  float4* Q;
  double* d[2];   // diagonal
  PairRot* rot;
  int n, np;
  GridBar gb;
};
__device__ __forceinline__ void pair_add(float& hi, float& lo, float x) {
  // two-sum of hi and x, then the low part: no contraction anywhere
  const float s = __fadd_rn(hi, x), bb = __fsub_rn(s, hi);
  const float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(x, bb));
  const float l = __fadd_rn(lo, e);
  hi = __fadd_rn(s, l);
  lo = __fsub_rn(l, __fsub_rn(hi, s));
}
__device__ __forceinline__ float4 pair_add(float4 a, float dx, float dy) {
  pair_add(a.x, a.y, dx);
  pair_add(a.z, a.w, dy);
  return a;
}
__device__ __forceinline__ float4 pair_from(double2 v) {
  const float xh = __double2float_rn(v.x), yh = __double2float_rn(v.y);
  return make_float4(xh, __double2float_rn(v.x - (double)xh), yh, __double2float_rn(v.y - (double)yh));
}
// A and Q to pairs (in place: 16 bytes either way), the diagonal apart
__global__ void k_pair_in(double2* A, double2* Q, int n, double* __restrict__ d) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)n * n) return;
  const double2 a = A[t];
  if (t % n == t / n) d[t / n] = a.x;
  ((float4*)A)[t] = pair_from(a);
  ((float4*)Q)[t] = pair_from(Q[t]);
}
__global__ void k_pair_out(const float4* Q, int64_t nn, double2* __restrict__ out) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nn) return;
  const float4 q = Q[t];
  out[t] = make_double2((double)q.x + (double)q.y, (double)q.z + (double)q.w);
}

constexpr int kPairThreads32 = 512;
__global__ void __launch_bounds__(kPairThreads32, 1) k_jacobi_pair_sweep(PairSweepArgs a) {
  extern __shared__ __align__(16) unsigned char jsm[];
  const int n = a.n, np = a.np, P = np / 2;
  PairRot* rot = (PairRot*)jsm;   // P
  int* pp = (int*)(rot + P);      // P
  int* pq = pp + P;               // P
  unsigned epoch = 0;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  const int Pe = P + (P & 1);     // folded triangle: Pe / 2 rows of Pe + 1
  const int nA = (Pe / 2) * (Pe + 1), nQ = n * P;
  for (int r = 0; r < np - 1; ++r) {
    const int cur = r & 1;
    const float4* A = a.A[cur];
    const double* d = a.d[cur];
    // a few rotations a block: they are long chains of FP64 operations
    for (int k = blockIdx.x + gridDim.x * threadIdx.x; k < P; k += nth) {
      int p = rr_player(k, r, np), q = rr_player(np - 1 - k, r, np);
      if (p > q) { const int t = p; p = q; q = t; }
      double c = 1.0;
      double2 s = make_double2(0, 0);
      if (p < n) {
        const double app = d[p];
        double dp = app;
        if (q < n) {
          const float4 v = A[(size_t)q * n + p];
          const double2 apq = make_double2((double)v.x + (double)v.y, (double)v.z + (double)v.w);
          const double aqq = d[q];
          jacobi_rotation<double>(apq, app, aqq, c, s);
          // J^H A J: the diagonal moves by t |A_pq| = Re(conj(s) A_pq) / c
          const double sh = (s.x * apq.x + s.y * apq.y) / c;
          dp = app - sh;
          a.d[cur ^ 1][q] = aqq + sh;
        }
        a.d[cur ^ 1][p] = dp;
      }
      PairRot o;
      const double s2 = s.x * s.x + s.y * s.y;
      o.c1 = (float)(-s2 / (1.0 + c));  // c - 1 without cancellation
      o.sx = (float)s.x;
      o.sy = (float)s.y;
      o.sxl = (float)(s.x - (double)o.sx);
      o.syl = (float)(s.y - (double)o.sy);
      a.rot[k] = o;
    }
    if (!grid_sync(a.gb, epoch)) return;
    for (int k = threadIdx.x; k < P; k += blockDim.x) {
      int p = rr_player(k, r, np), q = rr_player(np - 1 - k, r, np);
      if (p > q) { const int t = p; p = q; q = t; }
      pp[k] = p;
      pq[k] = q;
      // written by other blocks before the barrier: past the L1 cache
      const float* g = &a.rot[k].c1;
      rot[k] = PairRot{__ldcg(g), __ldcg(g + 1), __ldcg(g + 2), __ldcg(g + 3), __ldcg(g + 4)};
    }
    __syncthreads();
    float4* An = a.A[cur ^ 1];
    for (int t = tid; t < nA + nQ; t += nth) {
      if (t < nA) {
        // folded: row f holds column l = Pe - 1 - f (its k = 0 .. l), then l = f
        const int f = t / (Pe + 1), u = t - f * (Pe + 1);
        const int l = u < Pe - f ? Pe - 1 - f : f, k = u < Pe - f ? u : u - (Pe - f);
        if (l >= P) continue;  // (k <= l)
        const int pk = pp[k], qk = pq[k], pl = pp[l], ql = pq[l];
        if (pk >= n || pl >= n) continue;
        const bool vk = qk < n, vl = ql < n;
        if (k == l) {
          if (vk) An[(size_t)qk * n + pk] = An[(size_t)pk * n + qk] = make_float4(0.f, 0.f, 0.f, 0.f);
          continue;
        }
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 a00 = A[(size_t)pl * n + pk];
        const float4 a01 = vl ? A[(size_t)ql * n + pk] : z;
        const float4 a10 = vk ? A[(size_t)pl * n + qk] : z;
        const float4 a11 = (vk && vl) ? A[(size_t)ql * n + qk] : z;
        const PairRot rk = rot[k], rl = rot[l];
        // corrections d = A J - A by columns, then J^H (.) - (.) by rows
        auto col = [&](float4 x, float4 y, float2& dx, float2& dy) {
          dx.x = rl.c1 * x.x - (rl.sx * y.x + rl.sy * y.z);
          dx.y = rl.c1 * x.z - (rl.sx * y.z - rl.sy * y.x);
          dy.x = rl.c1 * y.x + (rl.sx * x.x - rl.sy * x.z);
          dy.y = rl.c1 * y.z + (rl.sx * x.z + rl.sy * x.x);
        };
        float2 d00, d01, d10, d11;
        col(a00, a01, d00, d01);
        col(a10, a11, d10, d11);
        auto row = [&](float4 x0, float2 e0, float4 x1, float2 e1, float2& o0, float2& o1) {
          const float2 u0 = make_float2(x0.x + e0.x, x0.z + e0.y), u1 = make_float2(x1.x + e1.x, x1.z + e1.y);
          o0.x = e0.x + (rk.c1 * u0.x - (rk.sx * u1.x - rk.sy * u1.y));
          o0.y = e0.y + (rk.c1 * u0.y - (rk.sx * u1.y + rk.sy * u1.x));
          o1.x = e1.x + (rk.c1 * u1.x + (rk.sx * u0.x + rk.sy * u0.y));
          o1.y = e1.y + (rk.c1 * u1.y + (rk.sx * u0.y - rk.sy * u0.x));
        };
        float2 y00, y01, y10, y11;
        row(a00, d00, a10, d10, y00, y10);
        row(a01, d01, a11, d11, y01, y11);
        auto put = [&](int i, int j, float4 v, float2 e) {
          v = pair_add(v, e.x, e.y);
          An[(size_t)j * n + i] = v;
          An[(size_t)i * n + j] = make_float4(v.x, v.y, -v.z, -v.w);
        };
        put(pk, pl, a00, y00);
        if (vl) put(pk, ql, a01, y01);
        if (vk) put(qk, pl, a10, y10);
        if (vk && vl) put(qk, ql, a11, y11);
      } else {
        const int e = t - nA;
        const int l = e / n, i = e - l * n;
        const int pl = pp[l], ql = pq[l];
        if (pl >= n || ql >= n) continue;
        const PairRot c = rot[l];
        float4* Qp = a.Q + (size_t)pl * n + i;
        float4* Qq = a.Q + (size_t)ql * n + i;
        const float4 q0 = *Qp, q1 = *Qq;
        // s with its low part: a systematic error of s would turn the column
        const float x0 = c.c1 * q0.x - ((c.sx * q1.x + c.sy * q1.z) + (c.sxl * q1.x + c.syl * q1.z));
        const float y0 = c.c1 * q0.z - ((c.sx * q1.z - c.sy * q1.x) + (c.sxl * q1.z - c.syl * q1.x));
        const float x1 = c.c1 * q1.x + ((c.sx * q0.x - c.sy * q0.z) + (c.sxl * q0.x - c.syl * q0.z));
        const float y1 = c.c1 * q1.z + ((c.sx * q0.z + c.sy * q0.x) + (c.sxl * q0.z + c.syl * q0.x));
        *Qp = pair_add(q0, x0, y0);
        *Qq = pair_add(q1, x1, y1);
      }
    }
    if (!grid_sync(a.gb, epoch)) return;
  }
}

// One sweep on A (n x n, FP64 in, destroyed) and Q (FP64 in, pairs out); A1 a second
// buffer, ws the diagonals and rotations (16-byte aligned to 8).
static void pair_sweep(System& s, DenseWs& w, double2* A, double2* A1, double2* Q, int n, char* ws,
                       cudaStream_t st) {
  unsigned* ctl = (unsigned*)w.ctl;
  PWH_CUDA(cudaMemsetAsync(ctl, 0, 3 * sizeof(unsigned), st));  // barrier words
  const int np = n + (n & 1), P = np / 2;
  PairSweepArgs a;
  a.A[0] = (float4*)A;
  a.A[1] = (float4*)A1;
  a.Q = (float4*)Q;
  a.d[0] = (double*)(((uintptr_t)ws + 15) & ~(uintptr_t)15);
  a.d[1] = a.d[0] + n;
  a.rot = (PairRot*)(a.d[1] + n);
  a.n = n;
  a.np = np;
  a.gb.count = ctl;
  a.gb.unused = ctl + 1;
  a.gb.abort = (int*)(ctl + 2);
  a.gb.err = device_error_word(s);
  k_pair_in<<<(unsigned)(((int64_t)n * n + 255) / 256), 256, 0, st>>>(A, Q, n, a.d[0]);
  PWH_LAUNCH_CHECK();
  const size_t smem = (size_t)P * (sizeof(PairRot) + 2 * sizeof(int));
  static std::once_flag once;
  std::call_once(once, [] {
    cudaFuncSetAttribute(k_jacobi_pair_sweep, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         (kJacobiMaxN / 2 + 1) * (int)(sizeof(PairRot) + 2 * sizeof(int)));
  });
  int dev = 0, nsm = 0, per_sm = 0;
  PWH_CUDA(cudaGetDevice(&dev));
  PWH_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  PWH_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_jacobi_pair_sweep, kPairThreads32, smem));
  const int64_t items = (int64_t)P * P / 2 + (int64_t)n * P;
  const int want = (int)std::max<int64_t>(1, std::min<int64_t>((items + 511) / 512, nsm));
  const int blocks = std::max(1, std::min(want, nsm * std::max(per_sm, 1)));
  void* args[] = {&a};
  PWH_CUDA(cudaLaunchCooperativeKernel((void*)k_jacobi_pair_sweep, blocks, kPairThreads32, args, smem, st));
  note_launch();
}

static size_t jacobi_ws_bytes(size_t nn, int n) {
  // FP64: A0, A1, Q0, Q1, G, the scaled matrix;  FP32: a0, a1, q0, q1;  diagonal d;
  // the refinement's per-index arrays
  return 6 * nn * sizeof(double2) + 4 * nn * sizeof(float2) + (size_t)n * sizeof(double) + 512 +
         refine_bytes(n);
}

void jacobi_eigh(System& s, DenseWs& w, const double2* H, int64_t ldh, int n, int nk,
                 double* theta, double2* C, cudaStream_t st, double2* Qkeep, int64_t ldk,
                 int warm_m0, bool polish, double tol32, double tol64) {
  if (n > kJacobiMaxN) throw Error{PWH_ERR_ARG, "subspace larger than the Jacobi limit"};
  const size_t nn = (size_t)n * n;
  ensure(w.jac, jacobi_ws_bytes(nn, n));
  double2* A0 = (double2*)w.jac.p;
  double2* A1 = A0 + nn;
  double2* Q0 = A1 + nn;
  double2* Q1 = Q0 + nn;
  double2* G = Q1 + nn;
  double2* Hs = G + nn;
  float2* a0 = (float2*)(Hs + nn);
  float2* a1 = a0 + nn;
  float2* q0 = a1 + nn;
  float2* q1 = q0 + nn;
  double* dg = (double*)(q1 + nn);
  if (!w.ctl) PWH_CUDA(cudaMalloc((void**)&w.ctl, 64));
  unsigned* ctl = (unsigned*)w.ctl;
  PWH_CUDA(cudaMemsetAsync(ctl, 0, 64, st));
  // The 16 control words of w.ctl:
  //   0-2   grid barrier of launch_jacobi (count, generation, abort)
  //   4-6   FP32 stage: result buffer index, sweeps, rounds logged
  //   8-9   FP64 stage: result buffer index, sweeps
  //   12    convergence flag of the grid-wide kernel (launch_jacobi)
  //   13    largest element, where the matrix is scaled (eig_exponent)
  int* out_buf = (int*)(ctl + 8);
  int* ob32 = (int*)(ctl + 4);
  const int gq = (int)std::min<int64_t>(1024, ((int64_t)nn + 255) / 256);
  const double2 one = make_double2(1, 0), zero = make_double2(0, 0);
  const bool warm = warm_m0 > 0 && Qkeep;
  double2* Q = Q0;
  // The first FP64 sweep in FP32 pairs needs the FP32 stage's basis, so the matrix
  // comes in a range where that works.
  const bool scaled = polish && n >= kRefineMinN;
  if (scaled) {
    k_eig_max<<<gq, 256, 0, st>>>(H, ldh, n, ctl + 13);
    PWH_LAUNCH_CHECK();
    k_eig_scale<<<gq, 256, 0, st>>>(H, ldh, n, ctl + 13, Hs);
    PWH_LAUNCH_CHECK();
    H = Hs;
    ldh = n;
  }
  {
    TimedScope ts(s, KF_JACOBI32, st);
    // ---- stage 1 (FP32): rotate the start to near-diagonal
    const double2* start = H;
    int64_t ld_start = ldh;
    // FP32-accurate n x n products of the warm start: on the tensor cores
    // (x3_gemm) above n = 512, where Newton-Schulz steps in FP64 arithmetic
    // follow, else on the FP32 pipe
    auto f32 = [&](bool cj, const double2* A, int64_t lda, const double2* B, double2* C) {
      if (n > 512)
        cgemm_f32(s, cj, n, n, n, one, A, lda, B, n, zero, C, n, st);
      else
        cgemm_f32_simt(s, cj, n, n, n, one, A, lda, B, n, zero, C, n, st);
    };
    if (warm) {
      // start in the previous eigenbasis: A = Qw^H H Qw (FP32 arithmetic suffices)
      k_warm_basis<<<gq, 256, 0, st>>>(Qkeep, ldk, warm_m0, n, Q1);
      PWH_LAUNCH_CHECK();
      f32(false, H, ldh, Q1, G);
      f32(true, Q1, n, G, A1);
      start = A1;
      ld_start = n;
    }
    // FP32 sweeps down to ~5 times FP32 rounding, so that one FP64 sweep (quadratic
    // convergence) usually finishes.  The whole matrix in one cluster's shared
    // memory when it fits, else through global memory.
    if (!jacobi32_tuned(s, w, start, ld_start, n, tol32, 30, Q0, n, dg, ob32, st)) {
      k_c64_to_c32<<<gq, 256, 0, st>>>(start, ld_start, n, a0);
      PWH_LAUNCH_CHECK();
      k_warm_basis<<<gq, 256, 0, st>>>(nullptr, 0, 0, n, Q0);  // identity
      PWH_LAUNCH_CHECK();
      k_c64_to_c32<<<gq, 256, 0, st>>>(Q0, n, n, q0);
      PWH_LAUNCH_CHECK();
      launch_jacobi<float>(s, w, a0, a1, q0, q1, n, tol32, 30, ob32, st);
      // the FP32 eigenvectors sit in q0 or q1 (ob32[0]): widen them to FP64
      k_select_buf<<<gq, 256, 0, st>>>(q0, q1, ob32, (int64_t)nn, Q0);
      PWH_LAUNCH_CHECK();
      k_diag_of<float><<<(n + 255) / 256, 256, 0, st>>>(a0, a1, ob32, n, dg);
      PWH_LAUNCH_CHECK();
    }
    if (warm) {
      f32(false, Q1, n, Q0, A0);  // Qw Q32
      Q = A0;
    }
    if (!polish) {
      // reduced-precision result: one Newton-Schulz step towards the nearest
      // unitary, Q (3I - Q^H Q)/2 in FP32 arithmetic; eigenvalues as Rayleigh
      // quotients q^H H q of those vectors (the FP32 diagonal drifts by the
      // accumulated non-unitarity of FP32 rotations, about n sweeps x 1e-7)
      // (above n = 512 the FP32 GEMMs' own rounding, ~sqrt(n) FP32 units,
      // would exceed the FP32 basis' deviation: the step then runs on the
      // FP64-equivalent GEMM)
      double2* Qo = (Q == Q0) ? A0 : Q0;
      auto g3 = [&](bool cj, const double2* A, int64_t lda, const double2* B, double2* C) {
        if (n > 512)
          cgemm<double>(s, cj, n, n, n, one, A, lda, B, n, zero, C, n, st);
        else
          cgemm_f32_simt(s, cj, n, n, n, one, A, lda, B, n, zero, C, n, st);
      };
      g3(true, Q, n, Q, G);
      k_ns_rhs<<<gq, 256, 0, st>>>(G, n, A1);
      PWH_LAUNCH_CHECK();
      g3(false, Q, n, A1, Qo);
      g3(false, H, ldh, Qo, G);
      k_rayleigh<<<n, 128, 0, st>>>(Qo, G, n, dg);
      PWH_LAUNCH_CHECK();
      const int sb = (int)std::min<int64_t>(64, ((int64_t)nn + 1023) / 1024);
      k_select_eig<<<sb, 1024, n * sizeof(int), st>>>(dg, Qo, n, nk, theta, C, Qkeep, ldk);
      PWH_LAUNCH_CHECK();
      return;
    }
  }
  TimedScope ts(s, KF_JACOBI, st);
  // ---- stage 2 (FP64): exact unitary basis, A = Q^H H Q
  // Newton-Schulz to the nearest unitary: Q <- Q (3I - Q^H Q)/2, once in FP32
  // arithmetic, once in FP64
  double2* Qo = (Q == Q0) ? A0 : Q0;
  cgemm_f32_simt(s, true, n, n, n, one, Q, n, Q, n, zero, G, n, st);
  k_ns_rhs<<<gq, 256, 0, st>>>(G, n, A1);
  PWH_LAUNCH_CHECK();
  cgemm_f32_simt(s, false, n, n, n, one, Q, n, A1, n, zero, Qo, n, st);
  // one FP64 step leaves ~(3/4) e^2 of the FP32 basis' deviation e from
  // unitary (e grows like sqrt(n) FP32 roundings): a second step above n = 512
  // (into the buffer of the FP32-stage vectors, Q0 or A0, free by now)
  if (n > 512) {
    cgemm<double>(s, true, n, n, n, one, Qo, n, Qo, n, zero, G, n, st);
    k_ns_rhs<<<gq, 256, 0, st>>>(G, n, A1);
    PWH_LAUNCH_CHECK();
    double2* Qn = (Qo == Q0) ? A0 : Q0;
    cgemm<double>(s, false, n, n, n, one, Qo, n, A1, n, zero, Qn, n, st);
    Qo = Qn;
  }
  cgemm<double>(s, true, n, n, n, one, Qo, n, Qo, n, zero, G, n, st);
  k_ns_rhs<<<gq, 256, 0, st>>>(G, n, A1);
  PWH_LAUNCH_CHECK();
  cgemm<double>(s, false, n, n, n, one, Qo, n, A1, n, zero, Q1, n, st);   // Q1: unitary basis
  cgemm<double>(s, false, n, n, n, one, H, ldh, Q1, n, zero, G, n, st);
  cgemm<double>(s, true, n, n, n, one, Q1, n, G, n, zero, A0, n, st);    // A0 = Q^H H Q
  hermitize(A0, n, 0, n, st);
  PWH_CUDA(cudaMemcpyAsync(Q0, Q1, nn * sizeof(double2), cudaMemcpyDeviceToDevice, st));
  if (n < kRefineMinN) {
    // ---- stage 3 (FP64): polish sweeps on the nearly diagonal matrix.  Inside
    // a cluster of (nearly) equal eigenvalues the FP32 basis leaves an
    // unstructured block of FP32-rounding size that the polish diagonalises
    // from scratch, at linear convergence (about a factor 2.3 a sweep on
    // 128-fold degenerate levels), hence the allowance of 30 sweeps; a
    // warm-started Rayleigh-Ritz matrix needs two or three.
    launch_jacobi<double>(s, w, A0, A1, Q0, Q1, n, tol64, 30, out_buf, st);
  } else {
    // ---- stage 3 by products: one Jacobi sweep (which also fixes the phases
    // of the eigenvectors, to the third order of its angles), two refinement
    // steps, the target test with a last step, and Jacobi sweeps again only
    // where the target was missed.  The limits leave X unitary to 1e-15 in
    // clusters too, where angles up to them keep being applied.
    pair_sweep(s, w, A0, A1, Q0, n, (char*)(dg + n) + (((size_t)n * 56 + 64 + 15) & ~(size_t)15), st);
    k_pair_out<<<(unsigned)((nn + 255) / 256), 256, 0, st>>>((const float4*)Q0, (int64_t)nn, Q1);
    PWH_LAUNCH_CHECK();
    const RefineWs rw = refine_carve(dg + n, n);
    double2 *X = Q1, *Gx = A0, *S = A1, *Gr = Q0, *Xn = G;
    const unsigned g1 = (unsigned)((n + 255) / 256);
    static std::once_flag once;
    std::call_once(once, [] {
      cudaFuncSetAttribute(k_refine_m, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           kJacobiMaxN * (int)sizeof(double2));
    });
    const double lims[3] = {1e-3, 1e-6, 3e-8};
    for (int step = 0; step < 3; ++step) {
      cgemm<double>(s, false, n, n, n, one, H, ldh, X, n, zero, Gx, n, st);
      cgemm<double>(s, true, n, n, n, one, X, n, Gx, n, zero, S, n, st);
      hermitize(S, n, 0, n, st);
      cgemm<double>(s, true, n, n, n, one, X, n, X, n, zero, Gr, n, st);
      k_refine_diag<<<g1, 256, 0, st>>>(S, Gr, n, rw);
      PWH_LAUNCH_CHECK();
      k_refine_max<<<1, 1024, 0, st>>>(n, rw);
      PWH_LAUNCH_CHECK();
      k_refine_best<<<n, 128, 0, st>>>(S, Gr, n, rw);
      PWH_LAUNCH_CHECK();
      k_refine_pairs<<<g1, 256, 0, st>>>(S, Gr, n, lims[step], tol64, rw);
      PWH_LAUNCH_CHECK();
      k_refine_m<<<n, 128, n * sizeof(double2), st>>>(S, Gr, n, lims[step], step == 2, rw, Gx);
      PWH_LAUNCH_CHECK();
      cgemm<double>(s, false, n, n, n, one, X, n, Gx, n, zero, Xn, n, st);
      std::swap(X, Xn);
    }
    launch_jacobi<double>(s, w, S, Gr, X, Xn, n, tol64, 30, out_buf, st, rw.done, rw.mx + 1);
    A0 = S;
    A1 = Gr;
    Q0 = X;
    Q1 = Xn;
    G = Gx;
  }
  k_diag_of<double><<<(n + 255) / 256, 256, 0, st>>>(A0, A1, out_buf, n, dg);
  PWH_LAUNCH_CHECK();
  if (scaled) {
    k_eig_unscale<<<(n + 255) / 256, 256, 0, st>>>(dg, n, ctl + 13);
    PWH_LAUNCH_CHECK();
  }
  k_select_buf64<<<gq, 256, 0, st>>>(Q0, Q1, out_buf, (int64_t)nn, G);
  PWH_LAUNCH_CHECK();
  const int sb = (int)std::min<int64_t>(64, ((int64_t)nn + 1023) / 1024);
  k_select_eig<<<sb, 1024, n * sizeof(int), st>>>(dg, G, n, nk, theta, C, Qkeep, ldk);
  PWH_LAUNCH_CHECK();
}

void jacobi_reserve(DenseWs& w, int nmax, int kmax) {
  const size_t nn = (size_t)nmax * nmax;
  ensure(w.jac, jacobi_ws_bytes(nn, nmax));
  // the blocked Cholesky's scratch: two k x k complex FP64 matrices and the
  // per-column words (the FP32 factorisation needs less)
  ensure(w.chol, 2 * (size_t)kmax * kmax * sizeof(double2) + (size_t)kmax * 16 + 256);
  ensure(w.ns, (size_t)4 * kmax * kmax * sizeof(double2) + 64);
  // rotation logs and buffers of the kernels for n <= 512, the block
  // kernel's tiles above
  const int nsmall = std::min(nmax, 512);
  if (nsmall >= 64) {
    ensure(w.jlog, jacobi32_log_bytes(nsmall, 30));
    ensure(w.jlog, pj_log_bytes(nsmall, 30));
    ensure(w.pj, pj_buf_bytes(nsmall));
  }
  if (nmax > 512 && nmax <= kJacobiMaxN) ensure(w.pj, bj_buf_bytes(nmax));
  if (!w.ctl) PWH_CUDA(cudaMalloc((void**)&w.ctl, 64));
}

void hermitize(double2* H, int64_t ld, int m0, int m, cudaStream_t st) {
  if (m <= m0) return;
  int64_t tot = (int64_t)m * (m - m0);
  int blocks = (int)std::min<int64_t>(1024, (tot + 255) / 256);
  k_hermitize<<<blocks, 256, 0, st>>>(H, ld, m0, m);
  PWH_LAUNCH_CHECK();
}

// ---- Cholesky-QR factor over the whole GPU, for blocks too wide for one
// block's shared memory.  Same contract as k_cholqr.  The unit-diagonal
// Gram matrix goes to a k x k scratch (lower triangle, column-major); a
// right-looking Cholesky runs in panels of kCbw columns: each panel on one
// block (the pivot test and the column drops in column order, then the
// panel's own later columns), the trailing lower triangle updated by 32 x 32
// tiles over the whole GPU.  Dropped rows and columns become identity rows and
// columns, so that the inverse of the kept part is the inverse of the whole:
// the diagonal blocks are inverted first (one warp each), then every block
// column walks down its rows (one block each),
//     X_IJ = -X_II sum_{J <= M < I} L_IM X_MJ.
// The same operations as the one-block kernel in another summation order.
constexpr int kCbw = 32;

// keep[j] and dinv[j] = 1/sqrt(S_jj) from the diagonal (one block, k <= 1024)
__global__ void k_chol_diag(const double2* __restrict__ S, int k, const double* __restrict__ t0,
                            double drop_rel, int* __restrict__ keep, double* __restrict__ dinv) {
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    const double d = S[(size_t)j * k + j].x;
    const bool kp = d > 0.0 && (!t0 || sqrt(d) >= drop_rel * t0[j]);
    keep[j] = kp;
    dinv[j] = kp ? 1.0 / sqrt(d) : 0.0;
  }
}

// A = D^-1/2 S D^-1/2 on the lower triangle (upper triangle zero)
template <typename T>
__global__ void k_chol_scale(const double2* __restrict__ S, int k, const double* __restrict__ dinv,
                             cx<T>* __restrict__ A) {
  const int64_t tot = (int64_t)k * k;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % k), j = (int)(t / k);
    const double2 v = S[t];
    const double sc = dinv[i] * dinv[j];
    A[t] = i >= j ? mk<T>((T)(v.x * sc), (T)(v.y * sc)) : mk<T>((T)0, (T)0);
  }
}

// Columns [j0, j0 + nbp) of the factor, in order, on one block.
template <typename T>
__global__ void __launch_bounds__(1024) k_chol_panel(cx<T>* __restrict__ A, int k, int j0, int nbp,
                                                     int* __restrict__ keep, double piv_tol) {
  __shared__ T piv_s;
  __shared__ int keep_s;
  const int j1 = min(k, j0 + nbp);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int j = j0; j < j1; ++j) {
    if (threadIdx.x == 0) {
      const T piv = A[(size_t)j * k + j].x;
      int kp = keep[j];
      if (kp && !(piv > (T)piv_tol)) {
        kp = 0;
        keep[j] = 0;
      }
      keep_s = kp;
      piv_s = kp ? sqrt(piv) : (T)0;
      if (kp) A[(size_t)j * k + j] = mk<T>(piv_s, (T)0);
    }
    __syncthreads();
    if (keep_s) {
      const T rl = (T)1 / piv_s;
      for (int i = j + 1 + threadIdx.x; i < k; i += blockDim.x)
        A[(size_t)j * k + i] = scl<T>(A[(size_t)j * k + i], rl);
      __syncthreads();
      // the panel's later columns l, rows i >= l: a warp per column
      for (int l = j + 1 + warp; l < j1; l += nw) {
        const cx<T> alj = A[(size_t)j * k + l];
        for (int i = l + lane; i < k; i += 32)
          A[(size_t)l * k + i] = sub<T>(A[(size_t)l * k + i], mulc<T>(A[(size_t)j * k + i], alj));
      }
    }
    __syncthreads();
  }
}

// A[i][l] -= sum_{j0 <= j < j1, keep[j]} A[i][j] conj(A[l][j]) for j1 <= l <= i < k:
// 32 x 32 tiles of the trailing lower triangle, 256 threads with 2 x 2 outputs.
template <typename T>
__global__ void __launch_bounds__(256) k_chol_update(cx<T>* __restrict__ A, int k, int j0, int j1,
                                                     const int* __restrict__ keep) {
  const int ti = blockIdx.x, tl = blockIdx.y;
  if (ti < tl) return;
  const int i0 = j1 + ti * 32, l0 = j1 + tl * 32, nbp = j1 - j0;
  __shared__ cx<T> pi[32][kCbw + 1], pl[32][kCbw + 1];
  __shared__ int kp[kCbw];
  for (int t = threadIdx.x; t < 32 * nbp; t += blockDim.x) {
    const int r = t % 32, c = t / 32;
    const int i = i0 + r, l = l0 + r;
    pi[r][c] = i < k ? A[(size_t)(j0 + c) * k + i] : mk<T>((T)0, (T)0);
    pl[r][c] = l < k ? A[(size_t)(j0 + c) * k + l] : mk<T>((T)0, (T)0);
  }
  for (int c = threadIdx.x; c < nbp; c += blockDim.x) kp[c] = keep[j0 + c];
  __syncthreads();
  const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
  cx<T> acc[2][2];
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) acc[a][b] = mk<T>((T)0, (T)0);
  for (int c = 0; c < nbp; ++c) {
    if (!kp[c]) continue;
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int b = 0; b < 2; ++b)
        acc[a][b] = add<T>(acc[a][b], mulc<T>(pi[tx + 16 * a][c], pl[ty + 16 * b][c]));
  }
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int i = i0 + tx + 16 * a, l = l0 + ty + 16 * b;
      if (i < k && l < k && i >= l) {
        cx<T>* e = A + (size_t)l * k + i;
        *e = sub<T>(*e, acc[a][b]);
      }
    }
}

// dropped indices become identity rows and columns of the lower triangle
template <typename T>
__global__ void k_chol_sanitize(cx<T>* __restrict__ A, int k, const int* __restrict__ keep) {
  const int64_t tot = (int64_t)k * k;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % k), j = (int)(t / k);
    if (i < j || (keep[i] && keep[j])) continue;
    A[t] = mk<T>(i == j ? (T)1 : (T)0, (T)0);
  }
}

// X_II = L_II^-1 for the diagonal 32 x 32 blocks (one warp each; indices past
// k act as identity): lane c solves column c by forward substitution.
template <typename T>
__global__ void k_chol_inv_diag(const cx<T>* __restrict__ A, int k, cx<T>* __restrict__ X) {
  __shared__ cx<T> Ls[32][33], Xs[32][33];
  const int b0 = blockIdx.x * 32, lane = threadIdx.x;
  for (int c = 0; c < 32; ++c) {
    const int i = b0 + lane, j = b0 + c;
    Ls[lane][c] = (i < k && j < k) ? A[(size_t)j * k + i] : mk<T>(i == j ? (T)1 : (T)0, (T)0);
  }
  __syncwarp();
  for (int i = 0; i < 32; ++i) {
    cx<T> acc = mk<T>(i == lane ? (T)1 : (T)0, (T)0);
    for (int m = lane; m < i; ++m) acc = sub<T>(acc, mul<T>(Ls[i][m], Xs[m][lane]));
    Xs[i][lane] = i < lane ? mk<T>((T)0, (T)0) : scl<T>(acc, (T)1 / Ls[i][i].x);
  }
  __syncwarp();
  for (int c = 0; c < 32; ++c) {
    const int i = b0 + lane, j = b0 + c;
    if (i < k && j < k) X[(size_t)j * k + i] = Xs[lane][c];
  }
}

// The off-diagonal blocks of X = L^-1, one block column J per thread block
// (32 x 32 threads, thread (r, c) owns row r, column c of each block), rows
// of blocks in order: Y = sum_{J <= M < I} L_IM X_MJ, then X_IJ = -X_II Y.
template <typename T>
__global__ void __launch_bounds__(1024) k_chol_inv_cols(const cx<T>* __restrict__ A, int k,
                                                        cx<T>* __restrict__ X) {
  __shared__ cx<T> Ys[32][33];
  const int J = blockIdx.x, nbk = (k + 31) / 32;
  const int r = threadIdx.x % 32, c = threadIdx.x / 32;
  const int jcol = J * 32 + c;
  for (int I = J + 1; I < nbk; ++I) {
    const int irow = I * 32 + r;
    cx<T> y = mk<T>((T)0, (T)0);
    if (irow < k && jcol < k)
      for (int m = J * 32; m < I * 32; ++m)
        y = add<T>(y, mul<T>(A[(size_t)m * k + irow], X[(size_t)jcol * k + m]));
    Ys[r][c] = y;
    __syncthreads();
    cx<T> x = mk<T>((T)0, (T)0);
    if (irow < k && jcol < k)
      for (int q = 0; q < 32 && I * 32 + q < k; ++q)
        x = sub<T>(x, mul<T>(X[(size_t)(I * 32 + q) * k + irow], Ys[q][c]));
    if (irow < k && jcol < k) X[(size_t)jcol * k + irow] = x;
    // this block's new X_IJ is read by the next rows of blocks
    __syncthreads();
  }
}

__global__ void k_chol_rank(const int* __restrict__ keep, int k, int* __restrict__ rank,
                            int* __restrict__ kk) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    int c = 0;
    for (int j = 0; j < k; ++j) rank[j] = keep[j] ? c++ : -1;
    *kk = c;
  }
}

// Tr = D^-1/2 L^-H on the kept set: column rank(j), row i <= j holds
// conj((L^-1)_ji) / sqrt(S_ii) (Tr zeroed before)
template <typename T>
__global__ void k_chol_out(const cx<T>* __restrict__ X, int k, const int* __restrict__ keep,
                           const int* __restrict__ rank, const double* __restrict__ dinv,
                           double2* __restrict__ Tr) {
  const int64_t tot = (int64_t)k * k;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % k), j = (int)(t / k);
    if (i > j || !keep[i] || !keep[j]) continue;
    const cx<T> v = X[(size_t)i * k + j];
    Tr[(size_t)rank[j] * k + i] = make_double2((double)v.x * dinv[i], -(double)v.y * dinv[i]);
  }
}

template <typename T>
static void cholqr_blocked(DenseWs& w, const double2* S, int k, const double* t0, double drop_rel,
                           double piv_tol, double2* Tr, int* kk, cudaStream_t st) {
  const size_t kk2 = (size_t)k * k;
  ensure(w.chol, 2 * kk2 * sizeof(cx<T>) + (size_t)k * (2 * sizeof(int) + sizeof(double)) + 256);
  cx<T>* A = (cx<T>*)w.chol.p;
  cx<T>* X = A + kk2;
  double* dinv = (double*)(X + kk2);
  int* keep = (int*)(dinv + k);
  int* rank = keep + k;
  const int g = (int)std::min<int64_t>(2048, ((int64_t)kk2 + 255) / 256);
  k_chol_diag<<<1, 1024, 0, st>>>(S, k, t0, drop_rel, keep, dinv);
  PWH_LAUNCH_CHECK();
  k_chol_scale<T><<<g, 256, 0, st>>>(S, k, dinv, A);
  PWH_LAUNCH_CHECK();
  for (int j0 = 0; j0 < k; j0 += kCbw) {
    const int j1 = std::min(k, j0 + kCbw);
    k_chol_panel<T><<<1, 1024, 0, st>>>(A, k, j0, j1 - j0, keep, piv_tol);
    PWH_LAUNCH_CHECK();
    if (j1 < k) {
      const int nt = (k - j1 + 31) / 32;
      k_chol_update<T><<<dim3(nt, nt), 256, 0, st>>>(A, k, j0, j1, keep);
      PWH_LAUNCH_CHECK();
    }
  }
  k_chol_sanitize<T><<<g, 256, 0, st>>>(A, k, keep);
  PWH_LAUNCH_CHECK();
  const int nbk = (k + 31) / 32;
  k_chol_inv_diag<T><<<nbk, 32, 0, st>>>(A, k, X);
  PWH_LAUNCH_CHECK();
  k_chol_inv_cols<T><<<nbk, 1024, 0, st>>>(A, k, X);
  PWH_LAUNCH_CHECK();
  k_chol_rank<<<1, 32, 0, st>>>(keep, k, rank, kk);
  PWH_LAUNCH_CHECK();
  PWH_CUDA(cudaMemsetAsync(Tr, 0, kk2 * sizeof(double2), st));
  k_chol_out<T><<<g, 256, 0, st>>>(X, k, keep, rank, dinv, Tr);
  PWH_LAUNCH_CHECK();
}

template <typename T>
static void cholqr_launch(DenseWs& w, const double2* S, int k, const double* t0, double drop_rel,
                          double piv_tol, double2* Tr, int* kk, cudaStream_t st) {
  // the packed lower triangle in shared memory up to 192 KB (k = 156 in FP64,
  // 221 in FP32; the kernel's static arrays take the rest) on one block, else
  // the blocked factorisation over the whole GPU
  const size_t tri = (size_t)k * (k + 1) / 2 * sizeof(cx<T>);
  static std::once_flag attr_once;
  std::call_once(attr_once, [] {
    cudaFuncSetAttribute(k_cholqr<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 192 * 1024);
  });
  if (tri <= 192 * 1024) {
    k_cholqr<T, true><<<1, 1024, tri, st>>>(S, k, t0, drop_rel, piv_tol, nullptr, Tr, kk);
    PWH_LAUNCH_CHECK();
  } else {
    cholqr_blocked<T>(w, S, k, t0, drop_rel, piv_tol, Tr, kk, st);
  }
}

// ||S - I||_F^2 of the leading k x k block of S (ld lds), one block.
__global__ void k_dev_identity_f2(const double2* __restrict__ S, int64_t lds, int k,
                                  double* __restrict__ out) {
  __shared__ double red[32];
  double acc = 0.0;
  for (int64_t t = threadIdx.x; t < (int64_t)k * k; t += blockDim.x) {
    const int i = (int)(t % k), j = (int)(t / k);
    const double2 v = S[(size_t)j * lds + i];
    const double re = v.x - (i == j ? 1.0 : 0.0);
    acc += re * re + v.y * v.y;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double tot = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
    *out = tot;
  }
}
// dst (k x k, ld k) = leading k x k block of src (ld lds); identity when src is null
__global__ void k_copy_square(const double2* __restrict__ src, int64_t lds, int k,
                              double2* __restrict__ dst) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)k * k;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t % k), j = (int)(t / k);
    dst[t] = src ? src[(size_t)j * lds + i] : make_double2(i == j ? 1.0 : 0.0, 0.0);
  }
}

bool ns_inv_sqrt(System& s, DenseWs& w, const double2* S, int64_t lds, int k, bool fp64,
                 double2* Z, cudaStream_t st) {
  if (k < 1) return false;
  ensure(w.ns, (size_t)4 * k * k * sizeof(double2) + 64);
  if (!w.h_word) PWH_CUDA(cudaMallocHost((void**)&w.h_word, 64));
  double2* Y = (double2*)w.ns.p;
  double2* Zc = Y + (size_t)k * k;
  double2* M = Zc + (size_t)k * k;
  double2* Tm = M + (size_t)k * k;
  double* dev = (double*)(Tm + (size_t)k * k);
  k_dev_identity_f2<<<1, 1024, 0, st>>>(S, lds, k, dev);
  PWH_LAUNCH_CHECK();
  PWH_CUDA(cudaMemcpyAsync(w.h_word, dev, sizeof(double), cudaMemcpyDeviceToHost, st));
  PWH_CUDA(cudaStreamSynchronize(st));
  const double e0 = std::sqrt(w.h_word[0]);
  // coupled iteration: ||Z_j Y_j - I|| ~ (3/4) ||Z_{j-1} Y_{j-1} - I||^2
  if (!(e0 <= 1e-2)) return false;
  const int its = e0 <= 1e-4 ? 2 : 3;
  const int gq = (int)std::min<int64_t>(1024, ((int64_t)k * k + 255) / 256);
  k_copy_square<<<gq, 256, 0, st>>>(S, lds, k, Y);
  PWH_LAUNCH_CHECK();
  k_copy_square<<<gq, 256, 0, st>>>(nullptr, 0, k, Zc);
  PWH_LAUNCH_CHECK();
  const double2 one = make_double2(1, 0), zero = make_double2(0, 0);
  auto gemm = [&](const double2* A, const double2* B, double2* C) {
    if (fp64)
      cgemm<double>(s, false, k, k, k, one, A, k, B, k, zero, C, k, st);
    else
      cgemm_f32(s, false, k, k, k, one, A, k, B, k, zero, C, k, st);
  };
  for (int it = 0; it < its; ++it) {
    gemm(Zc, Y, Tm);                       // Z Y
    k_ns_rhs<<<gq, 256, 0, st>>>(Tm, k, M);  // M = (3I - Z Y) / 2
    PWH_LAUNCH_CHECK();
    gemm(Y, M, Tm);                        // Y <- Y M
    std::swap(Y, Tm);
    gemm(M, Zc, Tm);                       // Z <- M Z
    std::swap(Zc, Tm);
  }
  PWH_CUDA(cudaMemcpyAsync(Z, Zc, (size_t)k * k * sizeof(double2), cudaMemcpyDeviceToDevice, st));
  return true;
}

void cholqr_factor(System& s, DenseWs& w, const double2* S, int k, const double* t0,
                   double drop_rel, double2* Tr, int* kk, cudaStream_t st, bool fp32) {
  if (k > 1024) throw Error{PWH_ERR_ARG, "block of more than 1024 new directions"};
  TimedScope ts(s, KF_CHOLQR, st);
  // a pivot of the unit-diagonal Gram matrix below ~10x the rounding of its
  // arithmetic marks a numerically dependent column
  if (fp32)
    cholqr_launch<float>(w, S, k, t0, drop_rel, 1e-6, Tr, kk, st);
  else
    cholqr_launch<double>(w, S, k, t0, drop_rel, 1e-12, Tr, kk, st);
}

}  // namespace pwh

extern "C" pwh_status pwh_subspace_cholqr(pwh_system* sys, int32_t precision, int32_t k,
                                          const void* S, const double* t0, double drop_rel,
                                          void* Tr, int32_t* kept) {
  using namespace pwh;
  return guarded([&] {
    PWH_CHECK_ARG(sys && S && Tr && kept, "null argument");
    PWH_CHECK_ARG(k >= 1 && k <= 1024, "k out of range [1, 1024]");
    PWH_CHECK_ARG(precision == PWH_FP64 || precision == PWH_MIXED, "unknown precision");
    PWH_CHECK_ARG(std::isfinite(drop_rel) && drop_rel >= 0.0, "drop_rel must be >= 0");
    System& s = sys->s;
    DenseWs w;
    int* dk = nullptr;
    PWH_CUDA(cudaMalloc((void**)&dk, sizeof(int)));
    cholqr_factor(s, w, (const double2*)S, k, t0, drop_rel, (double2*)Tr, dk, s.stream,
                  precision != PWH_FP64);
    int h = 0;
    cudaError_t e = cudaMemcpyAsync(&h, dk, sizeof(int), cudaMemcpyDeviceToHost, s.stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s.stream);
    cudaFree(dk);
    PWH_CUDA(e);
    *kept = h;
  });
}

extern "C" pwh_status pwh_subspace_eigh(pwh_system* sys, int32_t n, const void* H, int64_t ldh,
                                        int32_t nk, double* theta, void* C, void* Q, int64_t ldq,
                                        int32_t warm, int32_t precision) {
  using namespace pwh;
  return guarded([&] {
    PWH_CHECK_ARG(sys && H && theta && C, "null argument");
    PWH_CHECK_ARG(n >= 1 && n <= kJacobiMaxN, "n out of range");
    PWH_CHECK_ARG(nk >= 1 && nk <= n, "nk out of range");
    PWH_CHECK_ARG(ldh >= n, "ldh < n");
    PWH_CHECK_ARG(!Q || ldq >= n, "ldq < n");
    PWH_CHECK_ARG(warm >= 0 && warm <= n && (warm == 0 || Q), "warm needs Q and 0 <= warm <= n");
    PWH_CHECK_ARG(precision == PWH_FP64 || precision == PWH_MIXED, "precision must be FP64 or MIXED");
    System& s = sys->s;
    static thread_local DenseWs* ws = nullptr;
    if (!ws) ws = new DenseWs();
    jacobi_eigh(s, *ws, (const double2*)H, ldh, n, nk, theta, (double2*)C, s.stream, (double2*)Q,
                ldq, warm, precision == PWH_FP64);
  });
}
