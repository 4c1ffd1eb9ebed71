// ibm_slice.cu -- the kernels of the barrier-free correction loop (see
// ibm_slice.cuh) and their launchers: the one-off build of the slices'
// lists, the correction, and the band collide+stream that follows it.
#include <algorithm>

#include "ibm_slice.cuh"

namespace ibm {

// ------------------------------------------------------------------ build
__device__ __forceinline__ unsigned int slice_hash(int key) { return (unsigned int)key * 2654435761u; }

// Finds key in an open-addressing table of `size` (a power of two) entries,
// inserting it if it is absent and *n is below cap; returns its slot, or -1
// when there is no room.  A new key takes the next index of *n.
__device__ __forceinline__ int table_insert(int* keys, unsigned short* vals, int size, int key, int* n, int cap,
                                            bool* fresh) {
  unsigned int h = slice_hash(key) >> 8;
  *fresh = false;
  for (int probe = 0; probe < size; ++probe, ++h) {
    const int at = (int)(h & (unsigned int)(size - 1));
    if (keys[at] == key) return at;
    if (keys[at] >= 0) continue;
    if (*(volatile int*)n >= cap) return -1;
    const int old = atomicCAS(&keys[at], -1, key);
    if (old == key) return at;
    if (old >= 0) continue;
    const int k = atomicAdd(n, 1);
    if (k >= cap) return -1;
    vals[at] = (unsigned short)k;
    *fresh = true;
    return at;
  }
  return -1;
}

// Index of a key that is in the table (0 if it is not).
__device__ __forceinline__ int table_find(const int* keys, const unsigned short* vals, int size, int key) {
  unsigned int h = slice_hash(key) >> 8;
  for (int probe = 0; probe < size; ++probe, ++h) {
    const int at = (int)(h & (unsigned int)(size - 1));
    if (keys[at] == key) return vals[at];
    if (keys[at] < 0) break;
  }
  return 0;
}

// The lists of one slice per CTA: the markers by depth (breadth first over
// the G rows), the nodes of their supports (owned ones first -- those whose
// lowest covering marker is one of the slice's own -- then the others of the
// depth <= 1 markers, then the rest) and the local copies of weights, rows
// and covering lists.  The order within a depth depends on the scheduling;
// every sum runs in list order over marker ids, so results do not.
// stat: [0] != 0 when a slice does not fit, [1], [2] largest node counts.
template <class R>
__global__ void __launch_bounds__(kSliceThreads) k_slice_build(SliceArgs<R> sl, int M, int N, const int* __restrict__ ctr,
                                                               const int* __restrict__ band_of,
                                                               const R* __restrict__ W, const int* __restrict__ bnode,
                                                               const int* __restrict__ bcnt,
                                                               const Ent<R>* __restrict__ ent,
                                                               const Ent<R>* __restrict__ G,
                                                               const int* __restrict__ gcnt, int* __restrict__ stat) {
  __shared__ int mkey[kSliceMarkHash], nkey[kSliceNodeHash];
  __shared__ unsigned short mval[kSliceMarkHash], nval[kSliceNodeHash];
  __shared__ int mid[kSliceMarkers];
  __shared__ int nm, nn, bad;
  constexpr int NT = kSliceThreads;
  const int s = blockIdx.x, t = threadIdx.x;
  int* head = sl.head + (size_t)s * kSliceHead;
  for (int k = t; k < kSliceMarkHash; k += NT) mkey[k] = -1;
  for (int k = t; k < kSliceNodeHash; k += NT) nkey[k] = -1;
  if (t == 0) { nm = 0; nn = 0; bad = ctr[CTR_ERR] & ~WARN_NOT_CONV; }   // a band that overflowed has no valid lists
  __syncthreads();
  const int m0 = s * sl.S, m1 = min(M, m0 + sl.S);
  auto add_marker = [&](int m) {
    bool fresh;
    const int at = table_insert(mkey, mval, kSliceMarkHash, m, &nm, kSliceMarkers, &fresh);
    if (at < 0) bad = 1;
    else if (fresh) mid[mval[at]] = m;
  };
  auto add_node = [&](int b) {
    bool fresh;
    const int at = table_insert(nkey, nval, kSliceNodeHash, b, &nn, kSliceNodes, &fresh);
    if (at < 0) bad = 1;
    else if (fresh) {
      const int k = nval[at];
      sl.nid[(size_t)s * kSliceNodes + k] = bnode[b];
      if (k < kSliceX1) sl.bid[(size_t)s * kSliceX1 + k] = b;
    }
  };
  for (int m = m0 + t; m < m1; m += NT) add_marker(m);
  __syncthreads();
  int lo = 0;
  for (int h = 0; h <= N; ++h) {
    const int hi = min(nm, kSliceMarkers);
    __syncthreads();
    if (t == 0) head[4 + h] = hi;
    if (h < N && !bad)
      for (int k = lo + t; k < hi; k += NT) {
        const int m = mid[k], c = gcnt[m];
        if (c > kSliceRow) { bad = 1; continue; }
        for (int j = 0; j < c; ++j) add_marker(G[(long long)m * kGCap + j].m);
      }
    lo = hi;
    __syncthreads();
  }
  const int nloc = min(nm, kSliceMarkers), d1 = N >= 1 ? head[5] : nloc, dj = N >= 1 ? head[4 + N - 1] : 0;
  // owned nodes, then those of the depth <= 1 markers, then all
  for (int pass = 0; pass < 3; ++pass) {
    const int mm = pass == 0 ? m1 - m0 : (pass == 1 ? d1 : nloc);
    if (!bad)
      for (int k = t; k < mm * kStencil; k += NT) {
        const int b = band_of[(long long)mid[k / kStencil] * kStencil + k % kStencil];
        if (b < 0) continue;
        if (pass == 0) {
          const int first = ent[(long long)b * kBandCap].m;
          if (first < m0 || first >= m1) continue;
        }
        add_node(b);
      }
    __syncthreads();
    if (t == 0) head[pass] = min(nn, kSliceNodes);
    __syncthreads();
  }
  const int nX1 = head[1], nX = head[2];
  if (t == 0) {
    head[3] = 0;
    if (nX1 > kSliceX1) bad = 1;
    atomicMax(&stat[1], nX);
    atomicMax(&stat[2], nX1);
  }
  __syncthreads();
  if (bad) {
    if (t == 0) atomicOr(&stat[0], 1);
    return;
  }
  // the markers' copies: thread t is local marker t in the correction kernel
  for (int k = t; k < nloc; k += NT) {
    const int m = mid[k];
    sl.mid[(size_t)s * kSliceMarkers + k] = m;
    unsigned int word = 0;
    for (int q = 0; q < kStencil; ++q) {
      const int b = band_of[(long long)m * kStencil + q];
      const unsigned int at = b < 0 ? 0u : (unsigned int)table_find(nkey, nval, kSliceNodeHash, b);
      sl.w[((size_t)s * kStencil + q) * kSliceMarkers + k] = b < 0 ? R(0) : W[(long long)m * kStencil + q];
      if (q & 1) sl.wi[((size_t)s * (kStencil / 2) + q / 2) * kSliceMarkers + k] = word | (at << 16);
      else word = at;
    }
    const int c = k < dj ? gcnt[m] : 0;
    sl.rn[(size_t)s * kSliceMarkers + k] = c;
    // at least kRowHead entries, padded with the marker itself at weight zero
    for (int j = 0; j < max(c, kRowHead); ++j) {
      const Ent<R> q = G[(long long)m * kGCap + min(j, max(c - 1, 0))];
      sl.rw[((size_t)s * kSliceRow + j) * kSliceMarkers + k] = j < c ? q.w : R(0);
      sl.ri[((size_t)s * kSliceRow + j) * kSliceMarkers + k] =
          (unsigned short)(j < c ? table_find(mkey, mval, kSliceMarkHash, q.m) : k);
    }
  }
  for (int k = t; k < nX1; k += NT) {
    const int b = sl.bid[(size_t)s * kSliceX1 + k];
    const int c = bcnt[b];
    if (c > kSliceEnt) atomicOr(&stat[0], 1);
    sl.en[(size_t)s * kSliceX1 + k] = min(c, kSliceEnt);
    for (int j = 0; j < min(c, kSliceEnt); ++j) {
      const Ent<R> q = ent[(long long)b * kBandCap + j];
      sl.ew[((size_t)s * kSliceEnt + j) * kSliceX1 + k] = q.w;
      sl.ei[((size_t)s * kSliceEnt + j) * kSliceX1 + k] =
          (unsigned short)table_find(mkey, mval, kSliceMarkHash, q.m);
    }
  }
}

// ------------------------------------------------------------------ correction
// rho and j of U band nodes at once: their 9 U loads are in flight together.
template <int P, int PAR, int U>
__device__ __forceinline__ void gather_nodes(const IbArgs<P>& a, const int (&n)[U], typename Prec<P>::R (&rho)[U],
                                             typename Prec<P>::R (&jx)[U], typename Prec<P>::R (&jy)[U]) {
  typedef typename Prec<P>::R R;
  typedef typename Prec<P>::S S;
  const Geom& g = a.g;
  S v[U][9];
  bool plain[U];
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int y = n[u] / g.nx, x = n[u] - y * g.nx;
    // away from the sides the locations are constant offsets
    plain[u] = PAR == 0 || (x > 0 && x < g.nx - 1 && y > 0 && y < g.ny - 1);
    const long long base = (long long)y * g.nxp + x;
    if (plain[u]) {
#pragma unroll
      for (int i = 0; i < 9; ++i)
        v[u][i] = PAR == 0 ? a.A[i * g.plane + base]
                           : a.A[opp(i) * g.plane + base - (long long)cy(i) * g.nxp - cx(i)];
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    R p[9];
    if (plain[u]) {
#pragma unroll
      for (int i = 0; i < 9; ++i) p[i] = Prec<P>::ld(v[u][i], PAR == 0 ? i : opp(i));
    } else {
      const int y = n[u] / g.nx, x = n[u] - y * g.nx;
      long long where;
#pragma unroll 1
      for (int i = 0; i < 9; ++i) p[i] = post_stream<P>(g, a.c, a.A, PAR, x, y, i, where);
    }
    moments9<R>(p, rho[u], jx[u], jy[u]);
  }
}

template <int P, int PAR>
__global__ void __launch_bounds__(kSliceThreads) k_ib_slice(IbArgs<P> a, SliceArgs<typename Prec<P>::R> sl) {
  typedef typename Prec<P>::R R;
  typedef typename Vec2<R>::T V;
  constexpr int NT = kSliceThreads;
  constexpr int U = sizeof(R) == 8 ? 1 : 2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = a.N;
  V* hist = reinterpret_cast<V*>(smem_raw);                  // [N + 1][kSliceMarkers] A^n
  R* nr = reinterpret_cast<R*>(hist + (size_t)(N + 1) * kSliceMarkers);   // [xmax] rho, jx, jy
  R* njx = nr + sl.xmax;
  R* njy = njx + sl.xmax;
  R* sxx = njy + sl.xmax;                                    // [x1max] sum_n j^n j^n
  R* sxy = sxx + sl.x1max;
  R* syy = sxy + sl.x1max;
  R* cm = syy + sl.x1max;                                    // [3][kSliceMarkers] C
  __shared__ R red[kSliceMaxCorr + 2][NT / 32];
  __shared__ int depth[kSliceMaxCorr + 2];                   // markers of depth <= h
  const int s = blockIdx.x, t = threadIdx.x, warp = t >> 5;
  const int* head = sl.head + (size_t)s * kSliceHead;
  const int nown = head[0], nX1 = head[1], nX = head[2];
  const int own = head[4], nloc = head[4 + N], d1 = head[5];
  const size_t sm = (size_t)s * kSliceMarkers;
  for (int k = t; k <= N; k += NT) depth[k] = head[4 + k];

  // the marker's weights are on their way while the nodes are gathered
  R w[kStencil];
  unsigned int wi[kStencil / 2];
  R ux = R(0), uy = R(0);
  if (t < nloc) {
#pragma unroll
    for (int q = 0; q < kStencil; ++q) w[q] = sl.w[((size_t)s * kStencil + q) * kSliceMarkers + t];
#pragma unroll
    for (int q = 0; q < kStencil / 2; ++q) wi[q] = sl.wi[((size_t)s * (kStencil / 2) + q) * kSliceMarkers + t];
    const int m = sl.mid[sm + t];
    ux = a.Ux[m];
    uy = a.Uy[m];
  }
  {
    const int* nid = sl.nid + (size_t)s * kSliceNodes;
    for (int k = t; k < nX; k += NT * U) {
      int n[U];
      R r[U], jx[U], jy[U];
#pragma unroll
      for (int u = 0; u < U; ++u) n[u] = nid[k + u * NT < nX ? k + u * NT : k];
      gather_nodes<P, PAR, U>(a, n, r, jx, jy);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u * NT < nX) {
          nr[k + u * NT] = r[u];
          njx[k + u * NT] = jx[u];
          njy[k + u * NT] = jy[u];
        }
    }
  }
  // the marker's G row
  R rw[kRowHead];
  unsigned short ri[kRowHead];
  int rn = 0;
  const int dj = N > 1 ? head[4 + N - 1] : 0;
  const int drow = max(dj, own);                             // r^N needs the owned rows
  if (t < drow) {
    rn = sl.rn[sm + t];
#pragma unroll
    for (int j = 0; j < kRowHead; ++j) {
      rw[j] = sl.rw[((size_t)s * kSliceRow + j) * kSliceMarkers + t];
      ri[j] = sl.ri[((size_t)s * kSliceRow + j) * kSliceMarkers + t];
    }
  }
  __syncthreads();

  // rho*, J*^0, b = A^1 (Eq. 22b, Eq. 28 in moment form)
  R rs = R(1), bx = R(0), by = R(0);
  R rmax = R(0);
  if (t < nloc) {
    R jx = R(0), jy = R(0);
    rs = R(0);
#pragma unroll
    for (int q = 0; q < kStencil; ++q) {
      const int k = (q & 1) ? (int)(wi[q / 2] >> 16) : (int)(wi[q / 2] & 0xffffu);
      rs += w[q] * nr[k];
      jx += w[q] * njx[k];
      jy += w[q] * njy[k];
    }
    bx = rs * ux - jx;
    by = rs * uy - jy;
    V z, b;
    z.x = z.y = R(0);
    b.x = bx;
    b.y = by;
    hist[t] = z;
    hist[kSliceMarkers + t] = b;
    if (t < own) rmax = (R)(sqrt(bx * bx + by * by) / rs);
  }
  if (warp * 32 < own) warp_max_to<R>(rmax, red[0]);
  __syncthreads();

  // A^{n+1} = A^n + b - G A^n, to depth N - n; r^n of the owned markers
  R ax = bx, ay = by;
  auto row = [&](const V* An, R& djx, R& djy) {
    R sx = R(0), sy = R(0);
#pragma unroll
    for (int j = 0; j < kRowHead; ++j) {
      const V v = An[ri[j]];
      sx += rw[j] * v.x;
      sy += rw[j] * v.y;
    }
    for (int j = kRowHead; j < rn; ++j) {
      const V v = An[sl.ri[((size_t)s * kSliceRow + j) * kSliceMarkers + t]];
      const R wj = sl.rw[((size_t)s * kSliceRow + j) * kSliceMarkers + t];
      sx += wj * v.x;
      sy += wj * v.y;
    }
    djx = bx - sx;
    djy = by - sy;
  };
  for (int n = 1; n <= N; ++n) {
    const V* An = hist + (size_t)n * kSliceMarkers;
    // the last pass only forms r^N
    const int active = n < N ? depth[N - n] : own;
    rmax = R(0);
    if (t < active) {
      R djx, djy;
      row(An, djx, djy);
      if (n < N) {
        ax = ax + djx;
        ay = ay + djy;
        V v;
        v.x = ax;
        v.y = ay;
        hist[(size_t)(n + 1) * kSliceMarkers + t] = v;
      }
      if (t < own) rmax = (R)(sqrt(djx * djx + djy * djy) / rs);
    }
    if (warp * 32 < own) warp_max_to<R>(rmax, red[n]);
    __syncthreads();
  }

  // per node of a depth <= 1 marker: sum_n j^n j^n; per owned node the summed
  // momentum correction D^N
  for (int k = t; k < nX1; k += NT) {
    const int cnt = sl.en[(size_t)s * kSliceX1 + k];
    R ew[8];
    unsigned short ei[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < cnt) {
        ew[j] = sl.ew[((size_t)s * kSliceEnt + j) * kSliceX1 + k];
        ei[j] = sl.ei[((size_t)s * kSliceEnt + j) * kSliceX1 + k];
      }
    const R j0x = njx[k], j0y = njy[k];
    R axx = R(0), axy = R(0), ayy = R(0);
    const int last = k < nown ? N : N - 1;
    for (int n = 0; n <= last; ++n) {
      const V* An = hist + (size_t)n * kSliceMarkers;
      R px = R(0), py = R(0);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        if (j < cnt) {
          const V v = An[ei[j]];
          px += ew[j] * v.x;
          py += ew[j] * v.y;
        }
      for (int j = 8; j < cnt; ++j) {
        const V v = An[sl.ei[((size_t)s * kSliceEnt + j) * kSliceX1 + k]];
        const R wj = sl.ew[((size_t)s * kSliceEnt + j) * kSliceX1 + k];
        px += wj * v.x;
        py += wj * v.y;
      }
      if (n < N) {
        const R jx = j0x + px, jy = j0y + py;
        axx += jx * jx;
        axy += jx * jy;
        ayy += jy * jy;
      } else {
        R* o = a.bq + 8 * (long long)sl.bid[(size_t)s * kSliceX1 + k];
        o[6] = px;
        o[7] = py;
      }
    }
    sxx[k] = axx;
    sxy[k] = axy;
    syy[k] = ayy;
  }
  __syncthreads();

  // C_l = N rho* U U - sum_x W_l(x) / rho(x) sum_n j^n j^n
  if (t < d1) {
    R pxx = R(0), pxy = R(0), pyy = R(0);
#pragma unroll
    for (int q = 0; q < kStencil; ++q) {
      const int k = (q & 1) ? (int)(wi[q / 2] >> 16) : (int)(wi[q / 2] & 0xffffu);
      const R v = w[q] / nr[k];
      pxx += v * sxx[k];
      pxy += v * sxy[k];
      pyy += v * syy[k];
    }
    cm[t] = R(N) * rs * ux * ux - pxx;
    cm[kSliceMarkers + t] = R(N) * rs * ux * uy - pxy;
    cm[2 * kSliceMarkers + t] = R(N) * rs * uy * uy - pyy;
  }
  __syncthreads();

  // Eq. 27 summed: the second-moment correction of the owned nodes
  for (int k = t; k < nown; k += NT) {
    const int cnt = sl.en[(size_t)s * kSliceX1 + k];
    R pxx = R(0), pxy = R(0), pyy = R(0);
    for (int j = 0; j < cnt; ++j) {
      const int m = sl.ei[((size_t)s * kSliceEnt + j) * kSliceX1 + k];
      const R wj = sl.ew[((size_t)s * kSliceEnt + j) * kSliceX1 + k];
      pxx += wj * cm[m];
      pxy += wj * cm[kSliceMarkers + m];
      pyy += wj * cm[2 * kSliceMarkers + m];
    }
    R* o = a.bq + 8 * (long long)sl.bid[(size_t)s * kSliceX1 + k];
    o[3] = pxx;
    o[4] = pxy;
    o[5] = pyy;
  }
  // A^N of the owned markers (the forces), the slice's residuals
  if (t < own) {
    V v;
    v.x = ax;
    v.y = ay;
    reinterpret_cast<V*>(a.Ah)[(long long)N * a.M + sl.mid[sm + t]] = v;
  }
  for (int n = t; n <= N; n += NT) {
    R m = R(0);
    for (int k = 0; k < (own + 31) / 32; ++k) m = nanmax(m, red[n][k]);
    sl.rpart[(size_t)s * (kSliceMaxCorr + 2) + n] = m;
  }
}

// ------------------------------------------------------------------ band collide
// One node of a band segment: corrected if it is a band node (its summed
// correction is ready in bq[3..7]), collided and streamed.  The nine loads
// need no look at the band map, so they are in flight with it; a step
// overwrites all nine slots that it reads, so the corrected populations stay
// in registers (rounded as the storage rounds them).  Nodes on a closed or
// open side go through the boundary rules.
template <int P, int PAR, bool MACRO, bool MRT>
__device__ __forceinline__ void finish_node(const IbArgs<P>& a, int x, int y) {
  typedef typename Prec<P>::R R;
  typedef typename Prec<P>::S S;
  const Geom& g = a.g;
  S* __restrict__ A = a.A;
  const bool special = PAR == 0 ? (x == 0 && g.bc[0] == BC_INLET) : needs_boundary_path(g, x, y);
  const int b = a.node2band[y * g.nx + x];
  if (special) {
    if (b >= 0) {
      const R* q = a.bq + 8 * (long long)b;
      for (int i = 0; i < 9; ++i) {
        long long where;
        const R v = post_stream<P>(g, a.c, A, PAR, x, y, i, where);
        (void)v;
        if (where < 0) continue;
        const int slot = (int)(where / g.plane);
        const R df = feq_i<R>(i, R(0), q[6], q[7], q[3], q[4], q[5]);
        A[where] = Prec<P>::st(Prec<P>::ld(A[where], slot) + df, slot);
      }
    }
    if (PAR == 0) even_node<P, MACRO, MRT>(g, a.c, A, a.mac, x, y);
    else odd_node<P, MACRO, MRT>(g, a.c, A, a.mac, x, y);
    return;
  }
  const int xm = x == 0 ? g.nx - 1 : x - 1, xp = x == g.nx - 1 ? 0 : x + 1;
  const int ym = y == 0 ? g.ny - 1 : y - 1, yp = y == g.ny - 1 ? 0 : y + 1;
  S v[9];
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int sx = PAR == 0 ? x : (cx(i) > 0 ? xm : (cx(i) < 0 ? xp : x));
    const int sy = PAR == 0 ? y : (cy(i) > 0 ? ym : (cy(i) < 0 ? yp : y));
    v[i] = A[(PAR == 0 ? i : opp(i)) * g.plane + (long long)sy * g.nxp + sx];
  }
  R p[9], ps[9], rho, jx, jy;
#pragma unroll
  for (int i = 0; i < 9; ++i) p[i] = Prec<P>::ld(v[i], PAR == 0 ? i : opp(i));
  if (b >= 0) {
    const R* q = a.bq + 8 * (long long)b;
    const R pxx = q[3], pxy = q[4], pyy = q[5], dx = q[6], dy = q[7];
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const int slot = PAR == 0 ? i : opp(i);
      const R df = feq_i<R>(i, R(0), dx, dy, pxx, pxy, pyy);
      p[i] = Prec<P>::ld(Prec<P>::st(p[i] + df, slot), slot);
    }
  }
  collide_full<P, MRT>(p, ps, rho, jx, jy, a.c);
  if (MACRO) write_macro<R>(a.mac, (long long)g.nx * g.ny, (long long)y * g.nx + x, rho, jx, jy);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int tx = PAR == 0 ? x : (cx(i) > 0 ? xp : (cx(i) < 0 ? xm : x));
    const int ty = PAR == 0 ? y : (cy(i) > 0 ? yp : (cy(i) < 0 ? ym : y));
    const int slot = PAR == 0 ? opp(i) : i;
    A[slot * g.plane + (long long)ty * g.nxp + tx] = Prec<P>::st(ps[i], slot);
  }
}

// Block 0 reduces the slices' residual maxima, the next nchunk blocks form
// the body forces (one chunk of kForceChunk markers each; the last to arrive
// adds the chunks up), the others collide and stream the 32-node row segments
// that hold band nodes, one warp per segment.  The forces are the longest
// chain in it: with one trip of loads per chunk, a halving tree for the FP64
// sums and the residuals in a block of their own it takes 10.8 us instead of
// 20.4 on a 300^2 lattice with 1029 markers (cold caches).
template <int P, int PAR, bool MACRO, bool MRT>
__global__ void __launch_bounds__(256) k_band_finish(IbArgs<P> a, SliceArgs<typename Prec<P>::R> sl) {
  typedef typename Prec<P>::R R;
  const int nchunk = (a.M + kForceChunk - 1) / kForceChunk, nfin = nchunk + 1;
  if (blockIdx.x == 0) {
    const int lane = threadIdx.x & 31;
    for (int n = threadIdx.x >> 5; n <= a.N; n += 8) {
      R m = R(0);
      for (int k = lane; k < sl.count; k += 32) m = nanmax(m, sl.rpart[(size_t)k * (kSliceMaxCorr + 2) + n]);
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) m = nanmax(m, __shfl_xor_sync(0xffffffffu, m, off));
      if (lane == 0) {
        a.resid[n] = m;
        if (n == a.N) ib_check_resid<P>(a);
      }
    }
    return;
  }
  if ((int)blockIdx.x < nfin) {
    __shared__ double sh[kChunkSumShared];
    __shared__ int last;
    ib_force_chunk<P>(a, a.Ah + (long long)a.N * 2 * a.M, blockIdx.x - 1, sh);
    if (nchunk > 1) {
      if (threadIdx.x == 0) {
        __threadfence();
        last = atomicAdd(sl.fin, 1) == nchunk - 1;
        if (last) *sl.fin = 0;                             // the next launch starts from zero
        __threadfence();
      }
      __syncthreads();
      if (!last) return;
    }
    ib_force_total<P>(a, 0, 1, sh);
    return;
  }
  const Geom& g = a.g;
  const int nseg = a.ctr[CTR_NSEG];
  const int lane = threadIdx.x & (kSegW - 1);
  const int nw = ((gridDim.x - nfin) * blockDim.x) / kSegW;
  for (int k = ((blockIdx.x - nfin) * blockDim.x + threadIdx.x) / kSegW; k < nseg; k += nw) {
    const int seg = a.seglist[k];
    const int y = seg / a.nseg_x, x = (seg - y * a.nseg_x) * kSegW + lane;
    if (x >= g.nx || nee_column(g, x)) continue;          // k_open_columns streams those
    finish_node<P, PAR, MACRO, MRT>(a, x, y);
  }
}

// ------------------------------------------------------------------ launchers
template <class R>
static SliceArgs<R> slice_args(const Ctx& h) {
  SliceArgs<R> s{};
  s.count = h.sl_count;
  s.S = h.sl_S;
  s.xmax = h.sl_xmax;
  s.x1max = h.sl_x1max;
  slice_bytes<R>(h.sl_count, (unsigned char*)h.sl_mem, &s);
  return s;
}

int slice_max_corr() { return kSliceMaxCorr; }

size_t slice_mem_bytes(int prec, int count) {
  return prec == PREC_FP64 ? slice_bytes<double>(count, nullptr, nullptr)
                           : slice_bytes<float>(count, nullptr, nullptr);
}

template <class R>
static cudaError_t slice_build_t(const Ctx& h, int* stat, cudaStream_t s) {
  SliceArgs<R> a = slice_args<R>(h);
  cudaError_t e = cudaMemsetAsync(a.fin, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  k_slice_build<R><<<h.sl_count, kSliceThreads, 0, s>>>(a, h.nm, h.desc.n_corr, h.dctr, h.dband_of, (const R*)h.dW,
                                                        h.dbnode, h.dbcnt, (const Ent<R>*)h.dent,
                                                        (const Ent<R>*)h.dG, h.dgcnt, stat);
  return cudaGetLastError();
}

cudaError_t launch_slice_build(const Ctx& h, int* stat, cudaStream_t s) {
  return h.r_bytes == 8 ? slice_build_t<double>(h, stat, s) : slice_build_t<float>(h, stat, s);
}

// Shared memory of the slice kernel for these local node counts, or 0 when
// the device cannot give it.
template <int P>
static size_t slice_smem_t(int N, int xmax, int x1max) {
  const size_t need = slice_smem_bytes<typename Prec<P>::R>(xmax, x1max, N);
  constexpr size_t kMax = 200 * 1024;
  if (need > kMax) return 0;
  if (cudaFuncSetAttribute(k_ib_slice<P, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMax) != cudaSuccess ||
      cudaFuncSetAttribute(k_ib_slice<P, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMax) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return need;
}

size_t slice_smem(int prec, int N, int xmax, int x1max) {
  switch (prec) {
    case PREC_FP64: return slice_smem_t<PREC_FP64>(N, xmax, x1max);
    case PREC_FP32: return slice_smem_t<PREC_FP32>(N, xmax, x1max);
    case PREC_FP16_DEV: return slice_smem_t<PREC_FP16_DEV>(N, xmax, x1max);
    default: return slice_smem_t<PREC_BF16_DEV>(N, xmax, x1max);
  }
}

template <int P>
static void slice_loop_t(const Ctx& h, int parity, bool macro, cudaStream_t s) {
  typedef typename Prec<P>::R R;
  IbArgs<P> a = make_ib_args<P>(h);
  SliceArgs<R> sl = slice_args<R>(h);
  const size_t smem = slice_smem_bytes<R>(sl.xmax, sl.x1max, a.N);
  const dim3 grid(sl.count), block(kSliceThreads);
  if (parity == 0) launch_prio_smem(k_ib_slice<P, 0>, grid, block, smem, s, h.ib_prio, a, sl);
  else launch_prio_smem(k_ib_slice<P, 1>, grid, block, smem, s, h.ib_prio, a, sl);
  const int nchunk = (h.nm + kForceChunk - 1) / kForceChunk;
  const int need = (h.segcap * kSegW + 255) / 256;
  const dim3 g2(1 + nchunk + std::max(1, std::min(need, 8 * h.ib_grid_max))), b2(256);
  auto go = [&](auto kern) { launch_prio(kern, g2, b2, s, h.ib_prio, a, sl); };
  if (a.c.mrt) {
    if (parity == 0) { if (macro) go(k_band_finish<P, 0, true, true>); else go(k_band_finish<P, 0, false, true>); }
    else { if (macro) go(k_band_finish<P, 1, true, true>); else go(k_band_finish<P, 1, false, true>); }
  } else {
    if (parity == 0) { if (macro) go(k_band_finish<P, 0, true, false>); else go(k_band_finish<P, 0, false, false>); }
    else { if (macro) go(k_band_finish<P, 1, true, false>); else go(k_band_finish<P, 1, false, false>); }
  }
}

void launch_slice_loop(const Ctx& h, int parity, bool macro, cudaStream_t s) {
  switch (h.prec) {
    case PREC_FP64: slice_loop_t<PREC_FP64>(h, parity, macro, s); break;
    case PREC_FP32: slice_loop_t<PREC_FP32>(h, parity, macro, s); break;
    case PREC_FP16_DEV: slice_loop_t<PREC_FP16_DEV>(h, parity, macro, s); break;
    default: slice_loop_t<PREC_BF16_DEV>(h, parity, macro, s); break;
  }
}

}  // namespace ibm
