// chol_cluster.cuh -- the damped GGN system's FP64 Cholesky factorisation
// (arXiv 2512.04579, Eq. 9) spread over a thread-block cluster, for batches
// that leave most SMs idle with one CTA per instance.
//
// One SM's FP64 pipe bounds the single-CTA factorisation (n^3 / 6 DFMA at
// 1.68 per clock: 0.38 ms of 0.78 at n = 200), and its one-warp diagonal
// steps most of the rest.  Here the lower matrix lives in the cluster's
// distributed shared memory as 16 x 16 blocks, whole block rows per CTA, and
// rank 0 runs the serial chain -- next panel block, next diagonal block, its
// factor and inverse -- one panel ahead of the other ranks' trailing update.
// Panels travel through distributed shared memory; two hardware cluster
// barriers separate a panel's phases (no spin waits).  The substitutions, the
// refinement residual and delta = S y run on the same block rows: the owner of
// a row block applies its inverted diagonal block, its 16 results go to every
// rank, one cluster barrier per panel.  Every entry sees the operations of
// chol.cuh and k_solve in the same order, so factor, step and iterates are
// bitwise those of the single-CTA kernel.
#pragma once
#include "chol.cuh"
#include "cluster_plan.cuh"

namespace gnm {

constexpr int kClThreads = 512;
static_assert(CNB == kClBlock, "the row plans count blocks of the panel width");

// The barriers below are .aligned: a warp's threads execute them together, so
// each first brings the warp's threads back together.
__device__ __forceinline__ void cl_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Barrier `id` of eight warps of the CTA.
__device__ __forceinline__ void bar_256(int id) {
  __syncwarp();
  asm volatile("bar.sync %0, 256;" ::"r"(id) : "memory");
}
__device__ __forceinline__ int cl_size() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int cl_my_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
// Doubles of dynamic shared memory this CTA was launched with.
__device__ __forceinline__ int64_t cl_dyn_words() {
  uint32_t r;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(r));
  return (int64_t)(r / 8);
}
// The shared-memory object that p is in this CTA, in the CTA of the given rank.
// A remote address is always this function's result or an index from it: one
// formed by adding a distance to a pointer into this CTA's shared memory would be
// stored to as this CTA's.
template <typename T>
__device__ __forceinline__ T* cl_map(T* p, int rank) {
  uint64_t q;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(q) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
  return reinterpret_cast<T*>(q);
}

// Shared memory of a cluster CTA, in doubles from a 16-byte aligned base.
// Blocks are stored column by column (entry (r, c) at 16 c + r).  Stores test
// their address against `words`, the CTA's dynamic shared memory, in the
// bounds-check build (has(); the CTAs of a cluster all have as much, so a store
// to another rank tests the address it was mapped from).
struct ClSmem {
  int64_t words;
  double* ybuf;  // [2][256] inverted diagonal blocks (row-major), by panel parity
  double* cbuf;  // [2][512] rank 0: blocks (p+1, p) and (p+1, p+1) of panel p, by parity
  double* lbuf;  // [256] rank 0: L of block (p+1, p)
  double* col;   // [2][34] rank 0: two columns of the diagonal factor, each with 1 / its pivot
  double* pbuf;  // [nblk][256] the panel's L blocks; after the factorisation the vectors (ClVec)
  double* blk;   // this rank's block rows: A, then L, with the inverse of the diagonal block in its place
  template <typename V>
  __device__ __forceinline__ bool has(const V* p) const {
    return GNM_IN(reinterpret_cast<const char*>(p) - reinterpret_cast<const char*>(ybuf), 8 * words - (int64_t)sizeof(V) + 1);
  }
};

// Vectors of n doubles that take the panel buffer's place (16 n doubles).
struct ClVec {
  double *rhs, *b, *z, *x, *dx, *s0, *delta;  // s0: two halves by panel parity
  float *yh, *yl;
  __device__ ClVec(double* p, int n)
      : rhs(p), b(p + n), z(p + 2 * n), x(p + 3 * n), dx(p + 4 * n), s0(p + 5 * n), delta(p + 7 * n),
        yh(reinterpret_cast<float*>(p + 8 * n)), yl(reinterpret_cast<float*>(p + 8 * n) + n) {}
};

struct ClusterChol {
  ClSmem m;
  const int* plan;   // [nblk]
  const int* rows;   // shared memory: this rank's block rows, ascending
  int* fail;         // shared memory [2]: failed diagonal blocks (cl_fail_word)
  int n, nblk, nrows, rank, size;
  bool rank0_rows;   // rank 0 owns block rows (and so needs the panels)

  // Blocks of L(I, p) = A(I, p) Y_p^T: 256 threads (t), thread (r, c) with the
  // column pairs dealt to the warps so that the four SM sub-partitions (warps
  // w and w + 4) get equally long dot products.  at: block A(I, p).
  __device__ __forceinline__ double panel_entry(const double* at, const double* Yp, int t, int& r, int& c) const {
    const int w = t >> 5, lane = t & 31;
    r = lane & 15;
    c = 2 * (w < 4 ? w : 11 - w) + (lane >> 4);
    double acc = 0.0;
#pragma unroll
    for (int q = 0; q < CNB; ++q)
      if (q <= c) acc = fma(at[q * 16 + r], Yp[c * 16 + q], acc);
    return acc;
  }

  // Step c of the diagonal factorisation on entry (r, k), k > c: col the scaled
  // column c, rj 1 / its pivot.
  static __device__ __forceinline__ double diag_step(double v, int r, int k, int c, double cr, double ck, double rj) {
    if (r >= k) return fma(-cr, ck, v);
    if (r <= c) return fma(-ck, r == c ? rj : cr, v);
    return v;
  }

  // Rank 0, threads t < 256: factor and invert diagonal block d, whose
  // reduced entries the caller holds (thread t: row r = t & 15, column k = t >> 4,
  // v = the entry for r >= k).  Threads above the diagonal (r < k) carry the
  // inverse's entry (k, r) instead: step c of the factorisation is also step c of
  // its accumulation, so a step costs one FP64 instruction per warp after the
  // pivot column, and that column (16 entries, L below and the inverse's row c
  // left of the pivot) sits in half a warp.  A warp holds two columns and
  // publishes both at once, so eight block barriers order the 16 columns.
  __device__ void diag(int d, double v) {
    const int t = threadIdx.x, r = t & 15, k = t >> 4, warp = t >> 5;
    const int nb = min(CNB, n - d * CNB);
    if (r < k) v = 0.0;
    bool ok = true;
    double rinv = 0.0;
    for (int w = 0; 2 * w < nb; ++w) {
      const int c0 = 2 * w, c1 = c0 + 1;
      double* col = m.col + (w & 1) * 34;
      if (warp == w) {
        double rj = pivot_rsqrt(__shfl_sync(0xffffffffu, v, c0), ok);
        if (k == c0) {
          v *= rj;
          if (m.has(col + r)) col[r] = v;
          if (r == c0) col[16] = rinv = rj;
        }
        if (c1 < nb) {
          const double cr = __shfl_sync(0xffffffffu, v, r), ck = __shfl_sync(0xffffffffu, v, c1);
          if (k == c1) v = diag_step(v, r, k, c0, cr, ck, rj);
          rj = pivot_rsqrt(__shfl_sync(0xffffffffu, v, 16 | c1), ok);
          if (k == c1) {
            v *= rj;
            if (m.has(col + 17 + r)) col[17 + r] = v;
            if (r == c1) col[33] = rinv = rj;
          }
        }
      }
      bar_256(1);
      if (k > c1) {
        v = diag_step(v, r, k, c0, col[r], col[k], col[16]);
        if (c1 < nb) v = diag_step(v, r, k, c1, col[17 + r], col[17 + k], col[33]);
      }
    }
    const double y = r < k ? v : (r == k ? rinv : 0.0);  // inverse entry (k, r)
    double* yd = m.ybuf + (d & 1) * 256 + k * CNB + r;
    if (m.has(yd)) {
#pragma unroll 4
      for (int q = 0; q < size; ++q) *cl_map(yd, q) = y;
    }
    if (!ok && (t & 31) == 0)
      for (int q = 0; q < size; ++q) *cl_map(fail + cl_fail_word(d), q) = 1;
  }

  // Rank 0, threads t < 256: from the buffered blocks of panel p, L of block
  // (p+1, p), then the next diagonal block's update, factor and inverse.
  __device__ void critical(int p) {
    const int t = threadIdx.x;
    const double* A1 = m.cbuf + (p & 1) * 512;
    int r, c;
    const double l = panel_entry(A1, m.ybuf + (p & 1) * 256, t, r, c);
    if (m.has(m.lbuf + c * 16 + r)) m.lbuf[c * 16 + r] = l;
    bar_256(1);
    r = t & 15;
    const int k = t >> 4;
    double v = 0.0;
    if (r >= k) {
      double acc = 0.0;
#pragma unroll
      for (int q = 0; q < CNB; ++q) acc = fma(m.lbuf[q * 16 + r], m.lbuf[q * 16 + k], acc);
      v = A1[256 + k * 16 + r] - acc;
    }
    diag(p + 1, v);
  }

  __device__ __forceinline__ double* block(int I, int K) const { return m.blk + ((int64_t)cl_slot(plan[I]) + K) * 256; }
  __device__ __forceinline__ bool own(int I) const { return cl_rank(plan[I]) == rank; }
  __device__ __forceinline__ void keep_inverse(int p) {
    if (own(p) && threadIdx.x < 256 && m.has(block(p, p) + threadIdx.x))
      block(p, p)[threadIdx.x] = m.ybuf[(p & 1) * 256 + threadIdx.x];
  }

  // Own rows' L blocks of panel p, in place and into every rank's panel buffer.
  __device__ void panel(int p) {
    const int t = threadIdx.x & 255, half = threadIdx.x >> 8;
    keep_inverse(p);
    for (int x = half; x < nrows; x += 2) {
      const int I = rows[x];
      if (I <= p) continue;
      int r, c;
      double* at = block(I, p);
      const double l = panel_entry(at, m.ybuf + (p & 1) * 256, t, r, c);
      double* pb = m.pbuf + I * 256 + c * 16 + r;
      if (m.has(pb)) {
#pragma unroll 4
        for (int q = rank0_rows ? 0 : 1; q < size; ++q) *cl_map(pb, q) = l;
      }
      bar_256(2 + half);  // the half's threads have read the block
      if (m.has(at + c * 16 + r)) at[c * 16 + r] = l;
    }
  }

  // Trailing update of own rows I >= p + 2 by panel p, 2 x 2 tiles per thread
  // (row p + 1 holds only the diagonal block that rank 0 updates).  Row p + 2,
  // updated first, also goes to rank 0 for the next panel's chain.
  __device__ void trailing(int p) {
    int x0 = 0;
    while (x0 < nrows && rows[x0] < p + 2) ++x0;
    int total = 0;
    for (int x = x0; x < nrows; ++x) total += rows[x] - p;
    double* next = rank == 0 ? m.cbuf : cl_map(m.cbuf, 0);
    for (int u = threadIdx.x; u < total * 64; u += kClThreads) {
      int b = u >> 6, x = x0;
      while (b >= rows[x] - p) b -= rows[x++] - p;
      const int I = rows[x], K = p + 1 + b;
      const int r0 = ((u >> 3) & 7) * 2, k0 = (u & 7) * 2;
      if (K == I && k0 > r0) continue;  // above the diagonal
      const double* la = m.pbuf + I * 256 + r0;
      const double* lb = m.pbuf + K * 256 + k0;
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll 4
      for (int c = 0; c < CNB; ++c) {
        const double2 av = *reinterpret_cast<const double2*>(la + c * 16);
        const double2 bv = *reinterpret_cast<const double2*>(lb + c * 16);
        acc[0][0] = fma(av.x, bv.x, acc[0][0]);
        acc[0][1] = fma(av.x, bv.y, acc[0][1]);
        acc[1][0] = fma(av.y, bv.x, acc[1][0]);
        acc[1][1] = fma(av.y, bv.y, acc[1][1]);
      }
      double* o = block(I, K) + k0 * 16 + r0;
      double2 e0 = *reinterpret_cast<double2*>(o), e1 = *reinterpret_cast<double2*>(o + 16);
      e0.x -= acc[0][0];
      e0.y -= acc[1][0];
      e1.x -= acc[0][1];
      e1.y -= acc[1][1];
      if (m.has(reinterpret_cast<double2*>(o + 16))) {
        *reinterpret_cast<double2*>(o) = e0;
        *reinterpret_cast<double2*>(o + 16) = e1;
      }
      if (I == p + 2) {
        const int at = ((p + 1) & 1) * 512 + (K - (p + 1)) * 256 + k0 * 16 + r0;
        double* w = next + at;
        if (m.has(reinterpret_cast<double2*>(m.cbuf + at + 16))) {
          *reinterpret_cast<double2*>(w) = e0;
          *reinterpret_cast<double2*>(w + 16) = e1;
        }
      }
    }
  }

  // Factorises the system that `entry(row, col)` gives (lower triangle; both
  // triangles are kept in H for the refinement residual).  Cluster-wide; false,
  // uniformly, without a factor.
  template <class Entry>
  __device__ bool factor(double* H, const Entry& entry) {
    const int t = threadIdx.x;
    __syncthreads();  // every thread has read the last attempt's flags
    if (t == 0) fail[0] = fail[1] = 0;
    for (int x = 0; x < nrows; ++x) {
      const int I = rows[x];
      double* row = block(I, 0);
      const int per = (I + 1) * CNB;
      for (int u0 = t; u0 < per * CNB; u0 += 4 * kClThreads) {
        double h[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {  // loads first: the stores below could alias them
          const int u = u0 + q * kClThreads, r = u / per, c = u - r * per, i = I * CNB + r;
          h[q] = (r < CNB && i < n && c <= i) ? entry(i, c) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int u = u0 + q * kClThreads, r = u / per, c = u - r * per, i = I * CNB + r;
          if (r >= CNB) break;
          if (i < n && c <= i && GNM_IN((int64_t)i * n + c, (int64_t)n * n)) {
            H[(int64_t)i * n + c] = h[q];
            H[(int64_t)c * n + i] = h[q];
          }
          if (m.has(row + c * 16 + r)) row[c * 16 + r] = h[q];
        }
      }
    }
    double v = 0.0;
    if (rank == 0) {
      const int r = t & 15, k = (t >> 4) & 15;
      if (t < 256 && r >= k && r < n) v = entry(r, k);
      for (int u = t; u < 512; u += kClThreads) {  // blocks (1, 0) and (1, 1)
        const int i = CNB + (u & 15), c = ((u >> 8) * CNB) + ((u >> 4) & 15);
        if (m.has(m.cbuf + u)) m.cbuf[u] = (i < n && c <= i) ? entry(i, c) : 0.0;
      }
    }
    cl_arrive();
    cl_wait();
    if (rank == 0 && t < 256) diag(0, v);
    cl_arrive();
    cl_wait();
    if (fail[cl_fail_word(0)]) return false;
    for (int p = 0; p + 1 < nblk; ++p) {
      panel(p);
      cl_arrive();
      if (rank == 0 && t < 256) critical(p);
      cl_wait();
      trailing(p);
      cl_arrive();
      cl_wait();
      if (fail[cl_fail_word(p + 1)]) return false;
    }
    keep_inverse(nblk - 1);
    return true;
  }

  // Row block of this thread's half warp (-1: none): rows[x] on warp x & 15,
  // lanes 0-15 or (x >= 16) 16-31, so that up to four row blocks run on an SM
  // sub-partition each.  cluster_plan allows at most 32 per rank.
  __device__ __forceinline__ int my_row() const {
    const int x = (int)(threadIdx.x >> 5) + (threadIdx.x & 16);
    return x < nrows ? rows[x] : -1;
  }

  // sum_c a[c sa] b[c] over c < nb in order; a full panel's operands are loaded ahead of the chain
  static __device__ __forceinline__ double dot(const double* a, int sa, const double* b, int nb) {
    double acc = 0.0;
    if (nb == CNB) {
      double x[CNB], y[CNB];
#pragma unroll
      for (int c = 0; c < CNB; ++c) {
        x[c] = a[c * sa];
        y[c] = b[c];
      }
#pragma unroll
      for (int c = 0; c < CNB; ++c) acc = fma(x[c], y[c], acc);
    } else {
      for (int c = 0; c < nb; ++c) acc = fma(a[c * sa], b[c], acc);
    }
    return acc;
  }

  // out = (L L^T)^-1 v.b on every rank; v.b holds this rank's rows (chol.cuh's
  // chol_forward and chol_backward).  v.z: every rank's copy of the forward result.
  __device__ void substitute(const ClVec& v, double* out) {
    const int I = my_row(), r = threadIdx.x & 15, i = I * CNB + r;
    const bool live = I >= 0 && i < n;
    const unsigned hm = (threadIdx.x & 16) ? 0xffff0000u : 0x0000ffffu;
    for (int p = 0; p < nblk; ++p) {
      const int p0 = p * CNB, nb = min(CNB, n - p0);
      if (I == p) {
        const double z = dot(block(p, p) + r * CNB, 1, v.b + p0, nb);
        if (r < nb && m.has(v.z + i))
#pragma unroll 4
          for (int q = 0; q < size; ++q) cl_map(v.z, q)[i] = z;
      }
      cl_arrive();
      cl_wait();
      if (I > p) {
        const double s = dot(block(I, p) + r, 16, v.z + p0, nb);
        if (live && m.has(v.b + i)) v.b[i] -= s;
        __syncwarp(hm);
      }
    }
    if (live && m.has(v.b + i)) v.b[i] = v.z[i];
    __syncwarp();
    for (int p = nblk - 1; p >= 0; --p) {
      const int p0 = p * CNB, nb = min(CNB, n - p0);
      double* s = v.s0 + (p & 1) * n;
      if (own(p)) {  // uniform over the CTA
        if (I == p) {
          const double z = dot(block(p, p) + r, CNB, v.b + p0, nb);
          if (r < nb && m.has(out + i))
#pragma unroll 4
            for (int q = 0; q < size; ++q) cl_map(out, q)[i] = z;
        }
        __syncthreads();
        for (int j = threadIdx.x; j < p0; j += kClThreads) {
          const double d = dot(block(p, j >> 4) + (j & 15) * 16, 1, out + p0, nb);
          if (m.has(s + j)) cl_map(s, cl_rank(plan[j >> 4]))[j] = d;
        }
      }
      cl_arrive();
      cl_wait();
      if (I >= 0 && I < p) {
        if (m.has(v.b + i)) v.b[i] -= s[i];
        __syncwarp(hm);
      }
    }
  }

  // v.b = v.rhs - H x on this rank's rows, one row per thread, columns in
  // order; the next 16 columns' loads (L2) are in flight meanwhile, about as
  // long as 16 dependent DFMA take.
  __device__ void residual(const ClVec& v, const double* H) {
    const int I = my_row(), i = I * CNB + (int)(threadIdx.x & 15);
    if (I < 0 || i >= n) return;
    const double* h = H + i;
    double acc = 0.0, cur[16], nxt[16];
#pragma unroll
    for (int q = 0; q < 16; ++q) cur[q] = q < n ? h[(int64_t)q * n] : 0.0;
    for (int c = 0; c < n; c += 16) {
#pragma unroll
      for (int q = 0; q < 16; ++q) nxt[q] = c + 16 + q < n ? h[(int64_t)(c + 16 + q) * n] : 0.0;
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (c + q < n) acc = fma(cur[q], v.x[c + q], acc);
#pragma unroll
      for (int q = 0; q < 16; ++q) cur[q] = nxt[q];
    }
    if (m.has(v.b + i)) v.b[i] = v.rhs[i] - acc;
  }

  // S y for this thread's row (srow_dot's order), the row block's rows of S
  // fetched 16 columns at a time by the whole warp through the block row's own
  // storage (the factor is done with).  Call with whole warps; ld: row stride.
  __device__ __forceinline__ void row_step(const double s, const ClVec& v, int c, double* h, double*) const {
    h[0] = fma(s, v.x[c], h[0]);
  }
  __device__ __forceinline__ void row_step(const float s, const ClVec& v, int c, float* h, float* l) const {
    const int k = c < (n & ~3) ? c & 3 : 0;
    h[k] = fmaf(s, v.yh[c], h[k]);
    l[k] = fmaf(s, v.yl[c], l[k]);
  }
  template <typename TA>
  __device__ double row_dot(const ClVec& v, const TA* S, int64_t ld) {
    TA h[4] = {0, 0, 0, 0}, l[4] = {0, 0, 0, 0};
    const int lane = threadIdx.x & 31, r = lane & 15, x0 = threadIdx.x >> 5;
    for (int x = x0; x < nrows; x += 16) {  // the warp's one or two row blocks
      const int I = rows[x];
      TA* tile = reinterpret_cast<TA*>(block(I, 0));  // [16][16], column c of row q at c ^ q
      const bool mine = (x >= 16) == (lane >= 16);
      TA cur[8];
      auto fetch = [&](int c0) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int i = I * CNB + 2 * q + (lane >> 4), c = c0 + r;
          cur[q] = (i < n && c < n) ? S[(int64_t)i * ld + c] : (TA)0;
        }
      };
      fetch(0);
      for (int c0 = 0; c0 < n; c0 += 16) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int row = 2 * q + (lane >> 4);
          if (m.has(tile + row * 16 + (r ^ row))) tile[row * 16 + (r ^ row)] = cur[q];
        }
        fetch(c0 + 16);  // zeros past the last column
        __syncwarp();
        if (mine) {
#pragma unroll
          for (int q = 0; q < 16; ++q)
            if (c0 + q < n) row_step(tile[r * 16 + (q ^ r)], v, c0 + q, h, l);
        }
        __syncwarp();
      }
    }
    if constexpr (sizeof(TA) == 8) return h[0];
    else
      return (((double)h[0] + (double)h[1]) + ((double)h[2] + (double)h[3])) +
             (((double)l[0] + (double)l[1]) + ((double)l[2] + (double)l[3]));
  }
};

}  // namespace gnm
