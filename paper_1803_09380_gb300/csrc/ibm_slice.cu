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
// stat: [0] != 0 when a slice does not fit, [1], [2] largest node counts,
// [3] largest marker count, [4] most markers that cover a node, [5] band
// segments.
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
  if (s == 0 && t == 0) stat[5] = ctr[CTR_NSEG];
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
    atomicMax(&stat[3], nloc);
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
  int most = 0;
  for (int k = t; k < nX1; k += NT) {
    const int b = sl.bid[(size_t)s * kSliceX1 + k];
    const int c = bcnt[b];
    if (c > kSliceEnt) atomicOr(&stat[0], 1);
    most = max(most, c);
    sl.en[(size_t)s * kSliceX1 + k] = min(c, kSliceEnt);
    for (int j = 0; j < kSliceEnt; ++j) {                    // padded at weight zero
      Ent<R> q;
      q.w = R(0);
      if (j < c) q = ent[(long long)b * kBandCap + j];
      sl.ew[((size_t)s * kSliceEnt + j) * kSliceX1 + k] = q.w;
      sl.ei[((size_t)s * kSliceEnt + j) * kSliceX1 + k] =
          (unsigned short)(j < c ? table_find(mkey, mval, kSliceMarkHash, q.m) : 0);
    }
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((t & 31) == 0) atomicMax(&stat[4], min(most, kSliceEnt));
}

// ------------------------------------------------------------------ correction
// rho and j of U band nodes at once: their 9 U loads are in flight together.
// Away from the sides (and in the even step everywhere) the locations are
// constant offsets; false: some node needs the boundary rules instead.
template <int PAR>
__device__ __forceinline__ bool plain_node(const Geom& g, int x, int y) {
  return PAR == 0 || (x > 0 && x < g.nx - 1 && y > 0 && y < g.ny - 1);
}
template <int P, int PAR, int U>
__device__ __forceinline__ bool gather_nodes(const IbArgs<P>& a, const int (&n)[U], typename Prec<P>::R (&rho)[U],
                                             typename Prec<P>::R (&jx)[U], typename Prec<P>::R (&jy)[U]) {
  typedef typename Prec<P>::R R;
  typedef typename Prec<P>::S S;
  const Geom& g = a.g;
  S v[U][9];
  bool all = true;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int y = n[u] / g.nx, x = n[u] - y * g.nx;
    const bool plain = plain_node<PAR>(g, x, y);
    all = all && plain;
    const long long base = (long long)y * g.nxp + x;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      v[u][i] = S(0.0f);
      if (plain)
        v[u][i] = PAR == 0 ? a.A[i * g.plane + base]
                           : a.A[opp(i) * g.plane + base - (long long)cy(i) * g.nxp - cx(i)];
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    R p[9];
#pragma unroll
    for (int i = 0; i < 9; ++i) p[i] = Prec<P>::ld(v[u][i], PAR == 0 ? i : opp(i));
    moments9<R>(p, rho[u], jx[u], jy[u]);
  }
  return all;
}

__device__ __forceinline__ void copy16_async(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned int)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// The loop of ib_step_body by one CTA, for a moving boundary whose band did
// not fit the slice's lists this step, with its results where k_slice_stream
// looks for them.
template <int P, int PAR>
__device__ __noinline__ void slice_fallback(const IbArgs<P>& a, const SliceArgs<typename Prec<P>::R>& sl) {
  typedef typename Prec<P>::R R;
  ib_step_body<P, PAR, kSliceThreads>(a, 0, 1);
  __syncthreads();
  const int nband = min(a.ctr[CTR_NBAND], a.bcap), N = a.N;
  for (int b = threadIdx.x; b < nband; b += kSliceThreads) {
    R pxx = R(0), pxy = R(0), pyy = R(0);
    for (int j = 0; j < a.bcnt[b]; ++j) {
      const Ent<R> q = a.ent[(long long)b * kBandCap + j];
      pxx += q.w * a.Cm[3 * q.m];
      pxy += q.w * a.Cm[3 * q.m + 1];
      pyy += q.w * a.Cm[3 * q.m + 2];
    }
    R* o = a.bq + 8 * (long long)b;
    o[3] = pxx;
    o[4] = pxy;
    o[5] = pyy;
  }
  if (PAR == 1)
    for (int k = threadIdx.x; k < 2 * a.M; k += kSliceThreads)
      a.Ah[(long long)(N + 1) * 2 * a.M + k] = a.Ah[(long long)N * 2 * a.M + k];
  for (int n = threadIdx.x; n <= N; n += kSliceThreads)
    sl.rpart[(size_t)PAR * sl.count * (kSliceMaxCorr + 2) + n] = a.resid[n];
}

// MOVING: one slice holds every marker, its lists rebuilt by k_rebuild after
// every step.
template <int P, int PAR, bool MOVING>
__global__ void __launch_bounds__(kSliceThreads, 2) k_ib_slice(IbArgs<P> a, SliceArgs<typename Prec<P>::R> sl) {
  typedef typename Prec<P>::R R;
  typedef typename Vec2<R>::T V;
  constexpr int NT = kSliceThreads;
  constexpr bool F64 = sizeof(R) == 8;
  constexpr bool PAIRS = F64 && !MOVING;                     // few nodes: (node, n) pairs fill the warps
  constexpr int U = F64 ? 2 : 4;                             // nodes gathered at once per thread
  constexpr int kLevels = F64 ? 6 : 11;                                // iterates of the history read at once
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = a.N, LM = sl.lmax, XM = sl.xmax, X1M = sl.x1max, EM = sl.emax;
  const int SM = (sl.S + 3) & ~3;
  V* hist = reinterpret_cast<V*>(smem_raw);                  // [N + 1][LM] A^n
  V* djs = hist + (size_t)(N + 1) * LM;                      // [N + 1][SM] dj^n of the owned markers
  V* jn = djs + (size_t)(N + 1) * SM;                      // PAIRS: [N + 1][X1M] spread A^n
  R* nr = reinterpret_cast<R*>(jn + (PAIRS ? (size_t)(N + 1) * X1M : 0));   // [XM] rho, jx, jy
  R* njx = nr + XM;
  R* njy = njx + XM;
  R* sxx = njy + XM;                                         // [X1M] sum_n j^n j^n
  R* sxy = sxx + X1M;
  R* syy = sxy + X1M;
  R* cm = syy + X1M;                                         // [3][LM] C
  R* dv = cm + 3 * LM;                                       // [kStencil][LM] W_l(x) / rho(x)
  R* rso = dv + kStencil * LM;                                                  // [SM] rho* of the owned markers
  R* sew = rso + SM;                          // [EM][X1M] covering lists
  int* sen = reinterpret_cast<int*>(sew + (size_t)EM * X1M);
  int* sbid = sen + X1M;                                     // [X1M] band indices of the owned nodes
  unsigned short* sei = reinterpret_cast<unsigned short*>(sbid + X1M);
  unsigned short* dk = sei + (size_t)EM * X1M;               // [kStencil][LM] their nodes
  __shared__ typename AtomicBits<R>::U rmax[kSliceMaxCorr + 2];   // residual maxima, as bits
  __shared__ int depth[kSliceMaxCorr + 2];                   // markers of depth <= h
  const int s = blockIdx.x, t = threadIdx.x;
  const int* head = sl.head + (size_t)s * kSliceHead;
  const int nown = head[0], nX1 = head[1], nX = head[2];
  const int own = head[4], nloc = head[4 + N], d1 = head[5];
  const size_t sm = (size_t)s * kSliceMarkers;
  dependency_release();                                      // k_slice_stream starts beside this kernel
  if (MOVING && head[3]) {
    slice_fallback<P, PAR>(a, sl);
    return;
  }
#pragma unroll 1
  for (int k = t; k <= N; k += NT) {
    depth[k] = head[4 + k];
    rmax[k] = 0;
  }

  // the gather's loads first, then what later phases read: the covering
  // lists to shared memory, the marker's weights and G row to registers
  {
    const int* nid = sl.nid + (size_t)s * kSliceNodes;
    bool all = true;
#pragma unroll 1
    for (int k = t; k < nX; k += NT * U) {
      int n[U];
      R r[U], jx[U], jy[U];
#pragma unroll
      for (int u = 0; u < U; ++u) n[u] = nid[k + u * NT < nX ? k + u * NT : k];
      all = gather_nodes<P, PAR, U>(a, n, r, jx, jy) && all;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (k + u * NT < nX) {
          nr[k + u * NT] = r[u];
          njx[k + u * NT] = jx[u];
          njy[k + u * NT] = jy[u];
        }
    }
    if (!all) {                                              // this thread's nodes at the sides
#pragma unroll 1
      for (int k = t; k < nX; k += NT) {
        const int n = nid[k], y = n / a.g.nx, x = n - y * a.g.nx;
        if (plain_node<PAR>(a.g, x, y)) continue;
        R p[9];
        post_stream9<P>(a.g, a.c, a.A, PAR, x, y, p);
        moments9<R>(p, nr[k], njx[k], njy[k]);
      }
    }
  }
  {
    // a row of the lists per warp: EM of weights, EM of markers, the counts,
    // the band indices
#pragma unroll 1
    for (int j = t >> 5; j <= 2 * EM + 1; j += NT / 32) {
      const char* from;
      char* to;
      int bytes;
      if (j < EM) {
        from = (const char*)(sl.ew + ((size_t)s * kSliceEnt + j) * kSliceX1);
        to = (char*)(sew + (size_t)j * X1M);
        bytes = nX1 * (int)sizeof(R);
      } else if (j < 2 * EM) {
        from = (const char*)(sl.ei + ((size_t)s * kSliceEnt + j - EM) * kSliceX1);
        to = (char*)(sei + (size_t)(j - EM) * X1M);
        bytes = nX1 * (int)sizeof(short);
      } else {
        from = (const char*)((j == 2 * EM ? sl.en : sl.bid) + (size_t)s * kSliceX1);
        to = (char*)(j == 2 * EM ? sen : sbid);
        bytes = (j == 2 * EM ? nX1 : nown) * (int)sizeof(int);
      }
#pragma unroll 1
      for (int k = (t & 31) * 16; k < bytes; k += 512) copy16_async(to + k, from + k);
    }
  }
  R w[kStencil];
  unsigned int wi[kStencil / 2];
  R ux = R(0), uy = R(0);
  int mid = 0;
  if (t < nloc) {
#pragma unroll
    for (int q = 0; q < kStencil; ++q) w[q] = sl.w[((size_t)s * kStencil + q) * kSliceMarkers + t];
#pragma unroll
    for (int q = 0; q < kStencil / 2; ++q) wi[q] = sl.wi[((size_t)s * (kStencil / 2) + q) * kSliceMarkers + t];
    mid = sl.mid[sm + t];
    ux = a.Ux[mid];
    uy = a.Uy[mid];
  }
  R rw[kRowHead];
  unsigned short ri[kRowHead];
  int rn = 0;
  const int drow = max(N > 1 ? head[4 + N - 1] : 0, own);    // r^N needs the owned rows
  if (t < drow) {
    rn = sl.rn[sm + t];
#pragma unroll
    for (int j = 0; j < kRowHead; ++j) {
      rw[j] = sl.rw[((size_t)s * kSliceRow + j) * kSliceMarkers + t];
      ri[j] = sl.ri[((size_t)s * kSliceRow + j) * kSliceMarkers + t];
    }
  }
  copy_async_wait();
  __syncthreads();

  // rho*, J*^0, b = A^1 (Eq. 22b, Eq. 28 in moment form)
  R rs = R(1), bx = R(0), by = R(0);
  if (t < nloc) {
    R jx = R(0), jy = R(0);
    rs = R(0);
#pragma unroll
    for (int q = 0; q < kStencil; ++q) {
      const int k = (q & 1) ? (int)(wi[q / 2] >> 16) : (int)(wi[q / 2] & 0xffffu);
      rs += w[q] * nr[k];
      jx += w[q] * njx[k];
      jy += w[q] * njy[k];
      if (t < d1) {
        dv[q * LM + t] = w[q];
        dk[q * LM + t] = (unsigned short)k;
      }
    }
    bx = rs * ux - jx;
    by = rs * uy - jy;
    V z, b;
    z.x = z.y = R(0);
    b.x = bx;
    b.y = by;
    hist[t] = z;
    hist[LM + t] = b;
    if (t < own) {
      djs[t] = b;
      rso[t] = rs;
    }
  }
  __syncthreads();

  // A^{n+1} = A^n + b - G A^n, to depth N - n; dj^n of the owned markers (the
  // last pass only forms dj^N)
  R ax = bx, ay = by;
#pragma unroll 1
  for (int n = 1; n <= N; ++n) {
    const V* An = hist + (size_t)n * LM;
    if (t < (n < N ? depth[N - n] : own)) {
      R sx = R(0), sy = R(0);
#pragma unroll
      for (int j = 0; j < kRowHead; ++j) {
        const V v = An[ri[j]];
        sx += rw[j] * v.x;
        sy += rw[j] * v.y;
      }
#pragma unroll 1
      for (int j = kRowHead; j < rn; ++j) {
        const V v = An[sl.ri[((size_t)s * kSliceRow + j) * kSliceMarkers + t]];
        const R wj = sl.rw[((size_t)s * kSliceRow + j) * kSliceMarkers + t];
        sx += wj * v.x;
        sy += wj * v.y;
      }
      V dj;
      dj.x = bx - sx;
      dj.y = by - sy;
      if (t < own) djs[(size_t)n * SM + t] = dj;
      if (n < N) {
        ax = ax + dj.x;
        ay = ay + dj.y;
        V v;
        v.x = ax;
        v.y = ay;
        hist[(size_t)(n + 1) * LM + t] = v;
      }
    }
    __syncthreads();
  }

  // r^n = max |dj^n| / rho* of the owned markers.  FP32: an n per warp; FP64:
  // (n, marker) pairs fill the warps
  if (F64) {
#pragma unroll 1
    for (int k = t; k < (N + 1) * own; k += NT) {
      const int n = k / own, l = k - n * own;
      const V d = djs[(size_t)n * SM + l];
      AtomicBits<R>::max_bits(&rmax[n], nanmax(R(0), (R)(sqrt(d.x * d.x + d.y * d.y) / rso[l])));
    }
  } else {
#pragma unroll 1
    for (int n = t >> 5; n <= N; n += NT / 32) {
      unsigned int m = 0;
#pragma unroll 1
      for (int l = t & 31; l < own; l += 32) {
        const V d = djs[(size_t)n * SM + l];
        m = max(m, __float_as_uint(nanmax(0.0f, (float)(sqrt(d.x * d.x + d.y * d.y) / rso[l]))));
      }
      m = __reduce_max_sync(0xffffffffu, m);
      if ((t & 31) == 0) rmax[n] = m;
    }
  }
  // W_l(x) / rho(x) of the depth <= 1 markers, spread over all threads
#pragma unroll 1
  for (int k = t; k < kStencil * d1; k += NT) {
    const int at = k / d1 * LM + k % d1;
    dv[at] = dv[at] / nr[dk[at]];
  }

  // per node of a depth <= 1 marker: sum_n j^n j^n; per owned node the summed
  // momentum correction D^N
  if (PAIRS) {
    // (node, n) pairs fill the warps; the sums over n follow in order
#pragma unroll 1
    for (int k = t; k < (N + 1) * nX1; k += NT) {
      const int n = k / nX1, x = k - n * nX1;
      if (n == N && x >= nown) continue;
      const int cnt = sen[x];
      const V* An = hist + (size_t)n * LM;
      V p;
      p.x = p.y = R(0);
#pragma unroll 1
      for (int j = 0; j < cnt; ++j) {
        const R wj = sew[(size_t)j * X1M + x];
        const V v = An[sei[(size_t)j * X1M + x]];
        p.x += wj * v.x;
        p.y += wj * v.y;
      }
      jn[(size_t)n * X1M + x] = p;
    }
    __syncthreads();
  }
#pragma unroll 1
  for (int k = t; k < nX1; k += NT) {
    const R j0x = njx[k], j0y = njy[k];
    R axx = R(0), axy = R(0), ayy = R(0);
    R* o = a.bq + 8 * (long long)sbid[k < nown ? k : 0];
    if (PAIRS) {
#pragma unroll 1
      for (int n = 0; n < N; ++n) {
        const V p = jn[(size_t)n * X1M + k];
        const R jx = j0x + p.x, jy = j0y + p.y;
        axx += jx * jx;
        axy += jx * jy;
        ayy += jy * jy;
      }
      if (k < nown) {
        const V p = jn[(size_t)N * X1M + k];
        o[6] = p.x;
        o[7] = p.y;
      }
    } else {
      // kLevels iterates at a time: their loads are independent, and the list
      // is walked once
      const int cnt = sen[k];
#pragma unroll 1
      for (int n0 = 0; n0 <= N; n0 += kLevels) {
        V p[kLevels];
#pragma unroll
        for (int u = 0; u < kLevels; ++u) p[u].x = p[u].y = R(0);
#pragma unroll 1
        for (int j = 0; j < cnt; ++j) {
          const R wj = sew[(size_t)j * X1M + k];
          const V* An = hist + (size_t)n0 * LM + sei[(size_t)j * X1M + k];
#pragma unroll
          for (int u = 0; u < kLevels; ++u)
            if (n0 + u <= N) {
              const V v = An[(size_t)u * LM];
              p[u].x += wj * v.x;
              p[u].y += wj * v.y;
            }
        }
#pragma unroll
        for (int u = 0; u < kLevels; ++u) {
          if (n0 + u < N) {
            const R jx = j0x + p[u].x, jy = j0y + p[u].y;
            axx += jx * jx;
            axy += jx * jy;
            ayy += jy * jy;
          } else if (n0 + u == N && k < nown) {
            o[6] = p[u].x;
            o[7] = p[u].y;
          }
        }
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
#pragma unroll 4
    for (int q = 0; q < kStencil; ++q) {
      const int k = dk[q * LM + t];
      const R v = dv[q * LM + t];
      pxx += v * sxx[k];
      pxy += v * sxy[k];
      pyy += v * syy[k];
    }
    cm[t] = R(N) * rs * ux * ux - pxx;
    cm[LM + t] = R(N) * rs * ux * uy - pxy;
    cm[2 * LM + t] = R(N) * rs * uy * uy - pyy;
  }
  // A^N of the owned markers (the forces), the slice's residuals
  if (t < own) {
    V v;
    v.x = ax;
    v.y = ay;
    reinterpret_cast<V*>(a.Ah)[(long long)(N + PAR) * a.M + mid] = v;
  }
#pragma unroll 1
  for (int n = t; n <= N; n += NT)
    sl.rpart[((size_t)PAR * sl.count + s) * (kSliceMaxCorr + 2) + n] = AtomicBits<R>::from_bits(rmax[n]);
  __syncthreads();

  // Eq. 27 summed: the second-moment correction of the owned nodes
#pragma unroll 1
  for (int k = t; k < nown; k += NT) {
    const int cnt = sen[k];
    R pxx = R(0), pxy = R(0), pyy = R(0);
#pragma unroll 1
    for (int j = 0; j < cnt; ++j) {
      const int m = sei[(size_t)j * X1M + k];
      const R wj = sew[(size_t)j * X1M + k];
      pxx += wj * cm[m];
      pxy += wj * cm[LM + m];
      pyy += wj * cm[2 * LM + m];
    }
    R* o = a.bq + 8 * (long long)sbid[k];
    o[3] = pxx;
    o[4] = pxy;
    o[5] = pyy;
  }
}

// ------------------------------------------------------------------ band collide
// One node of a band segment: corrected if it is a band node (its summed
// correction is ready in bq[3..7]), collided and streamed.  The nine loads
// need no look at the band map, so they are in flight with it; a step
// overwrites all nine slots that it reads, so the corrected populations stay
// in registers (rounded as the storage rounds them).  Nodes on a closed or
// open side go through the boundary rules.
// WAIT: the correction comes from the kernel launched before.
template <int P, int PAR, bool MACRO, bool MRT, bool WAIT>
__device__ __forceinline__ void finish_node(const IbArgs<P>& a, int x, int y) {
  typedef typename Prec<P>::R R;
  typedef typename Prec<P>::S S;
  const Geom& g = a.g;
  S* __restrict__ A = a.A;
  const int b = a.node2band[y * g.nx + x];
  if (PAR == 1 && needs_boundary_path(g, x, y)) {
    if (WAIT) dependency_wait();
    if (b >= 0) {
      const R* q = a.bq + 8 * (long long)b;
#pragma unroll
      for (int i = 0; i < 9; ++i) {
        int sx = x, sy = y, slot = i, ws;
        if (!locE(g, x, y, i, sx, sy, slot, ws)) continue;
        S* at = A + slot_index(g, slot, sx, sy);
        const R df = feq_i<R>(i, R(0), q[6], q[7], q[3], q[4], q[5]);
        *at = Prec<P>::st(Prec<P>::ld(*at, slot) + df, slot);
      }
    }
    odd_boundary<P, MACRO, MRT>(g, a.c, A, a.mac, x, y);
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
  if (WAIT) dependency_wait();
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
  if (PAR == 0 && x == 0 && g.bc[0] == BC_INLET) {             // as even_node
#pragma unroll
    for (int i = 0; i < 9; ++i) ps[i] = a.c.feq_in[i];
    rho = a.c.rho0; jx = a.c.rho0 * a.c.inlet_u[0]; jy = a.c.rho0 * a.c.inlet_u[1];
  }
  if (MACRO) write_macro<R>(a.mac, (long long)g.nx * g.ny, (long long)y * g.nx + x, rho, jx, jy);
#pragma unroll
  for (int i = 0; i < 9; ++i) {
    const int tx = PAR == 0 ? x : (cx(i) > 0 ? xp : (cx(i) < 0 ? xm : x));
    const int ty = PAR == 0 ? y : (cy(i) > 0 ? yp : (cy(i) < 0 ? ym : y));
    const int slot = PAR == 0 ? opp(i) : i;
    A[slot * g.plane + (long long)ty * g.nxp + tx] = Prec<P>::st(ps[i], slot);
  }
}

// The residuals and body forces of the step whose correction ran with parity
// `par`, by block k0 of 1 + nchunk blocks of NT threads: block 0 reduces the
// slices' residual maxima, the others form the forces, one chunk of kForceChunk
// markers each; the last to arrive adds the chunks up.  WAIT: that correction
// is the kernel launched before (what does not depend on it is loaded before
// the wait).  store false: a later step's results, formed in the same launch,
// are the ones to keep.
template <int P, int NT, bool WAIT>
__device__ __forceinline__ void force_block(const IbArgs<P>& a, const SliceArgs<typename Prec<P>::R>& sl, int k0,
                                            int par, bool store, ForceShared<NT>& sh) {
  typedef typename Prec<P>::R R;
  const int nchunk = (a.M + kForceChunk - 1) / kForceChunk;
  if (k0 == 0) {
    if (WAIT) dependency_wait();
    const int lane = threadIdx.x & 31;
    const R* rp = sl.rpart + (size_t)par * sl.count * (kSliceMaxCorr + 2);
#pragma unroll 1
    for (int n = threadIdx.x >> 5; n <= a.N; n += NT / 32) {
      R m = R(0);
      for (int k = lane; k < sl.count; k += 32) m = nanmax(m, rp[(size_t)k * (kSliceMaxCorr + 2) + n]);
#pragma unroll
      for (int off = 16; off >= 1; off >>= 1) m = nanmax(m, __shfl_xor_sync(0xffffffffu, m, off));
      if (lane == 0) {
        if (store) a.resid[n] = m;
        if (n == a.N) ib_check_resid<P>(a, m);
      }
    }
    return;
  }
  double* fpart = a.fpart + (size_t)par * nchunk * a.nb * 3;
  ib_force_chunk<P, NT, WAIT>(a, a.Ah + (long long)(a.N + par) * 2 * a.M, k0 - 1, fpart, sh);
  if (nchunk > 1) {
    if (threadIdx.x == 0) {
      __threadfence();
      sh.last = atomicAdd(sl.fin + par, 1) == nchunk - 1;
      if (sh.last) sl.fin[par] = 0;                           // the next launch starts from zero
      __threadfence();
    }
    __syncthreads();
    if (!sh.last) return;
  }
  ib_force_total<P>(a, 0, 1, fpart, store);
}

// The 32-node row segments that hold band nodes, collided and streamed, one
// warp per segment, by block k0 of nblk.  WAIT: as above; the segments'
// populations are loaded before the wait.
template <int P, int PAR, bool MACRO, bool MRT, int NT, bool WAIT>
__device__ __forceinline__ void band_block(const IbArgs<P>& a, int k0, int nblk) {
  const Geom& g = a.g;
  const int nseg = a.ctr[CTR_NSEG];
  const int lane = threadIdx.x & (kSegW - 1);
  // blocks first, then their warps: few segments spread over all SMs
#pragma unroll 1
  for (int k = (threadIdx.x >> 5) * nblk + k0; k < nseg; k += nblk * (NT / 32)) {
    const int seg = a.seglist[k];
    const int y = seg / a.nseg_x, x = (seg - y * a.nseg_x) * kSegW + lane;
    if (x >= g.nx || nee_column(g, x)) continue;          // the extrapolation columns are streamed apart
    finish_node<P, PAR, MACRO, MRT, WAIT>(a, x, y);
  }
}

constexpr int kFinishThreads = kForceChunk;
template <int P, int PAR, bool MACRO, bool MRT>
__global__ void __launch_bounds__(kFinishThreads) k_band_finish(IbArgs<P> a, SliceArgs<typename Prec<P>::R> sl) {
  const int nfin = 1 + (a.M + kForceChunk - 1) / kForceChunk;
  __shared__ ForceShared<kFinishThreads> fs;
  if ((int)blockIdx.x < nfin) force_block<P, kFinishThreads, false>(a, sl, blockIdx.x, PAR, true, fs);
  else band_block<P, PAR, MACRO, MRT, kFinishThreads, false>(a, blockIdx.x - nfin, gridDim.x - nfin);
}

// Everything of a step but the correction, as one launch behind the slice
// kernel (programmatic dependent launch): rows of blocks with the edge nodes
// (odd step), the band-free spans and the extrapolation columns, which need
// nothing of the correction and run beside it, then the band segments, which
// wait for it.  Those come after three quarters of the lattice's rows: on a
// large lattice they then find the correction done (20 to 23 us into the 185 and
// 201 us, even and odd, of a 4096^2 FP32 step) instead of holding registers while
// they wait, and are not the launch's tail, where their dependent loads took 10
// us.  The correction releases this launch at its start: released after its
// gather, it ended earlier (17 against 21 us) but the step later (188 and 204 us
// against 185 and 201).  One stream and two launches a step, without
// fork, join or priorities.
//
// The forces are the longest chain behind the correction (5 us against 1.5
// for the band: two dependent FP64 sums with an arrival between them), so
// inside a graph of several steps each step's forces and residuals are formed
// in the next step's launch, off the chain; the graph's last step forms its own.
struct StepShape {
  int bx;                      // blocks per row
  int edge_rows, span_rows;    // rows of blocks: edge nodes, lattice rows
  int head_rows, tail_rows;    // lattice rows before the rows of the blocks below; those
  int open;                    // blocks of extrapolation columns,
  int fprev, fnow;             // of the previous and this step's forces (0: none),
  int nblk;                    // and of band segments
};
constexpr int kStepThreads = kK1Threads;
// As k_collide_stream, but 72 registers for the FP32 even step, whose spans
// spill at 64 beside the other blocks' code.
constexpr int step_min_blocks(int P, int PAR) {
  return P == PREC_FP32 && PAR == 0 ? 14 : k1_min_blocks(P, PAR);
}
template <int P, int PAR, bool MACRO, bool MRT>
__global__ void __launch_bounds__(kStepThreads, step_min_blocks(P, PAR))
    k_slice_stream(IbArgs<P> a, SliceArgs<typename Prec<P>::R> sl, const int* __restrict__ segflag, StepShape sh) {
  __shared__ ForceShared<kStepThreads> fs;
  int row = blockIdx.y;
  if (PAR == 1) {
    if (row < sh.edge_rows) {
      k1_edge_node<P, MACRO, K1_MAIN, MRT>(a.g, a.c, a.A, a.mac, segflag, a.nseg_x,
                                           ((long long)row * sh.bx + blockIdx.x) * kStepThreads + threadIdx.x);
      return;
    }
    row -= sh.edge_rows;
  }
  const bool tail = row >= sh.head_rows && row < sh.head_rows + sh.tail_rows;
  if (!tail) {
    if (row >= sh.head_rows) row -= sh.tail_rows;
    k1_span<P, PAR, MACRO, K1_MAIN, MRT>(a.g, a.c, a.A, a.mac, segflag, a.nseg_x, row,
                                         (blockIdx.x * kStepThreads + threadIdx.x) >> 5, threadIdx.x & 31);
    return;
  }
  int k = (row - sh.head_rows) * sh.bx + blockIdx.x;
  if (k < sh.open) {
    const int q = k * kStepThreads + threadIdx.x;
    if (q < 2 * a.g.ny) open_column<P, PAR, MACRO, MRT>(a.g, a.c, a.A, a.mac, q / a.g.ny, q % a.g.ny);
    return;
  }
  k -= sh.open;
  if (k < sh.fprev) {
    force_block<P, kStepThreads, false>(a, sl, k, PAR ^ 1, sh.fnow == 0, fs);
    return;
  }
  k -= sh.fprev;
  if (k < sh.fnow) {
    force_block<P, kStepThreads, true>(a, sl, k, PAR, true, fs);
    return;
  }
  k -= sh.fnow;
  if (k == 0) dependency_wait();                           // the launch ends after the correction in any case
  if (k < sh.nblk) band_block<P, PAR, MACRO, MRT, kStepThreads, true>(a, k, sh.nblk);
}

// ------------------------------------------------------------------ moving bodies
// After a step of a lattice with moving bodies, one CTA: the Newton-Euler
// update (Eqs. 37-42), the rigid motion of the markers, and the band and the
// lists of its single slice for the next step -- in one launch where the
// general path takes nine, each waiting for the one before, and builds the
// rows of G one marker to a thread (48 us of the 118 us of a step with two
// disks of 63 markers).  Here a warp finds the few markers that a marker
// couples with by their windows and forms their G_lm a lane each; weights are
// formed per axis (8 instead of 32 cosines a marker: FP64 issues at two lanes a
// clock).  Every number is formed by the expressions of the general path in the
// same order.  A band that does not fit (more nodes or covering markers than
// the lists hold, a periodic axis shorter than two windows) is built by the
// general path's items in the same CTA and flagged in head[3].
constexpr int kRebuildThreads = 1024;
template <class R>
struct RebuildArgs {
  Geom g;
  int M, nb, points, nseg_x, bcap, segcap, move;
  int xcap, ecap;                  // nodes and covering markers that the lists hold
  BodyDev* bodies;
  const int* mbody;
  const double *dX, *dY, *ds;
  double *X, *Y;
  R *Ux, *Uy;
  int *node2band, *bnode, *segflag, *seglist, *ctr;
  // the general path's arrays
  R* W;
  int *node_of, *claim, *band_of, *bcnt, *gcnt;
  Ent<R> *ent, *G;
};

// Shared memory of k_rebuild: weights of the stencil slots and their products
// with ds, the axis weights, node table, covering lists.
template <class R>
struct RebuildShared {
  double wx[2][4][kSliceMarkers];          // axis weights
  double cs[kSliceMarkers], sn[kSliceMarkers];   // of the bodies
  R w[kStencil][kSliceMarkers], wds[kStencil][kSliceMarkers];
  int key[kSliceNodeHash];
  unsigned short val[kSliceNodeHash];
  unsigned short at[kStencil][kSliceMarkers];    // local node, 0xffff: outside
  int node[kSliceX1], cnt[kSliceX1];
  unsigned short list[kSliceEnt][kSliceX1];      // marker * 16 + slot
  int bx[kSliceMarkers], by[kSliceMarkers];
  unsigned short cand[kSliceRow][kSliceMarkers]; // coupled markers, ascending
  int rows[kSliceMarkers];
  int nn, nseg, bad;
};

// Difference of two window origins on one axis, the shorter way round.
__device__ __forceinline__ int window_step(int d, int n, bool periodic) {
  if (periodic) {                                // bodies may be whole periods apart
    d %= n;
    if (d > n / 2) d -= n;
    else if (d < -(n / 2)) d += n;
  }
  return d;
}

template <class R>
__global__ void __launch_bounds__(kRebuildThreads) k_rebuild(RebuildArgs<R> a, SliceArgs<R> sl) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RebuildShared<R>& sh = *reinterpret_cast<RebuildShared<R>*>(smem_raw);
  constexpr int NT = kRebuildThreads;
  const Geom& g = a.g;
  const int t = threadIdx.x, M = a.M;
  const bool px = g.bc[0] == BC_PERIODIC, py = g.bc[2] == BC_PERIODIC;
  // (slot, marker) pairs: marker ml, slots mq, mq + mstep, ..
  const int mshift = M <= 64 ? 6 : (M <= 128 ? 7 : 8), mstep = NT >> mshift;
  const int ml = t & ((1 << mshift) - 1), mq = ml < M ? t >> mshift : 64;
  // the old band leaves the maps; the table is cleared
  const int nold = min(a.ctr[CTR_NBAND], a.bcap);
  for (int b = t; b < nold; b += NT) band_clear_item(g, a.bnode, a.node2band, a.segflag, a.nseg_x, b);
  for (int k = t; k < kSliceNodeHash; k += NT) sh.key[k] = -1;
  for (int k = t; k < a.xcap; k += NT) sh.cnt[k] = 0;
  if (t == 0) { sh.nn = 0; sh.nseg = 0; sh.bad = (px && g.nx < 8) || (py && g.ny < 8); }
  if (a.move) {
    body_update_cta(g, a.bodies, a.nb);
    if (t < a.nb) sincos(a.bodies[t].theta - a.bodies[t].theta0, &sh.sn[t], &sh.cs[t]);
  }
  __syncthreads();
  if (t == 0) { a.ctr[CTR_NBAND] = 0; a.ctr[CTR_NSEG] = 0; }
  if (t < M) {
    double X, Y;
    const int mb = a.mbody[t];
    const BodyDev& B = a.bodies[mb];
    if (a.move && B.kind != IBM_BODY_FIXED) {                // marker_move_item
      const double cs = sh.cs[mb], sn = sh.sn[mb];
      X = B.xc[0] + cs * a.dX[t] - sn * a.dY[t];
      Y = B.xc[1] + sn * a.dX[t] + cs * a.dY[t];
      a.X[t] = X;
      a.Y[t] = Y;
      a.Ux[t] = (R)(B.u[0] - B.omega * (Y - B.xc[1]));
      a.Uy[t] = (R)(B.u[1] + B.omega * (X - B.xc[0]));
    } else {
      X = a.X[t];
      Y = a.Y[t];
    }
    const int bx = (int)floor(X) - 1, by = (int)floor(Y) - 1;
    sh.bx[t] = bx;
    sh.by[t] = by;
    sh.wx[0][0][t] = X;
    sh.wx[1][0][t] = Y;
  }
  __syncthreads();
  // axis weights; each pass keeps the position in slot 0 until it is replaced
  double aw[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int k = t + q * NT;
    if (k < 8 * M) {
      const int l = k >> 3, ax = (k >> 2) & 1, i = k & 3;
      aw[q] = delta_w(a.points, sh.wx[ax][0][l] - (double)((ax ? sh.by[l] : sh.bx[l]) + i));
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int k = t + q * NT;
    if (k < 8 * M) sh.wx[(k >> 2) & 1][k & 3][k >> 3] = aw[q];
  }
  __syncthreads();
  // stencil weights, nodes
#pragma unroll 1
  for (int q = mq; q < kStencil; q += mstep) {
    const int l = ml;
    const int x = wrap_axis(sh.bx[l] + (q & 3), g.nx, px), y = wrap_axis(sh.by[l] + (q >> 2), g.ny, py);
    double w = 0.0;
    unsigned short at = 0xffff;
    if (x >= 0 && y >= 0) {
      w = sh.wx[0][q & 3][l] * sh.wx[1][q >> 2][l];
      bool fresh;
      const int slot = table_insert(sh.key, sh.val, kSliceNodeHash, y * g.nx + x, &sh.nn, a.xcap, &fresh);
      if (slot < 0) sh.bad = 1;
      else {
        at = (unsigned short)slot;                           // the value is complete after the barrier
        if (fresh) sh.node[sh.val[slot]] = y * g.nx + x;
      }
    }
    const R wr = (R)w;
    sh.w[q][l] = wr;
    sh.wds[q][l] = (R)((double)wr * a.ds[l]);
    sh.at[q][l] = at;
  }
  __syncthreads();
  const int nn = min(sh.nn, a.xcap);
  if (!sh.bad) {
    // covering lists: entries in any order, then by marker
#pragma unroll 1
    for (int q = mq; q < kStencil; q += mstep) {
      const int l = ml;
      if (sh.at[q][l] == 0xffff) continue;
      const int n = sh.val[sh.at[q][l]];
      sh.at[q][l] = (unsigned short)n;
      const int pos = atomicAdd(&sh.cnt[n], 1);
      if (pos < a.ecap) sh.list[pos][n] = (unsigned short)(l * kStencil + q);
      else sh.bad = 1;
    }
  }
  __syncthreads();
  // every thread's branch is settled before a warp below may find a row that is
  // too long: the barriers inside are met by all of them or by none
  const bool fits = !sh.bad;
  __syncthreads();
  if (fits) {
    for (int k = t; k < nn; k += NT) {
      const int c = sh.cnt[k], n = sh.node[k];
      for (int i = 1; i < c; ++i) {
        const unsigned short v = sh.list[i][k];
        int j = i - 1;
        while (j >= 0 && sh.list[j][k] > v) { sh.list[j + 1][k] = sh.list[j][k]; --j; }
        sh.list[j + 1][k] = v;
      }
      sl.nid[k] = n;
      sl.bid[k] = k;
      sl.en[k] = c;
      for (int j = 0; j < a.ecap; ++j) {
        const unsigned short v = j < c ? sh.list[j][k] : 0;
        sl.ew[(size_t)j * kSliceX1 + k] = j < c ? sh.wds[v % kStencil][v / kStencil] : R(0);
        sl.ei[(size_t)j * kSliceX1 + k] = (unsigned short)(v / kStencil);
      }
      a.bnode[k] = n;
      a.node2band[n] = k;
      const int y = n / g.nx, seg = y * a.nseg_x + (n - y * g.nx) / kSegW;
      if (atomicCAS(&a.segflag[seg], 0, 1) == 0) {
        const int at = atomicAdd(&sh.nseg, 1);
        if (at < a.segcap) a.seglist[at] = seg;
        else atomicOr(&a.ctr[CTR_ERR], ERR_SEG_CAP);
      }
    }
    // coupled markers: those whose windows share a node inside the domain
    const int warp = t >> 5, lane = t & 31;
#pragma unroll 1
    for (int l = warp; l < M; l += NT / 32) {
      const int bx = sh.bx[l], by = sh.by[l];
      int nc = 0;
#pragma unroll 1
      for (int m0 = 0; m0 < M; m0 += 32) {
        const int m = m0 + lane;
        bool near = false;
        if (m < M) {
          const int dx = window_step(sh.bx[m] - bx, g.nx, px), dy = window_step(sh.by[m] - by, g.ny, py);
          int x0 = bx + max(dx, 0), x1 = bx + min(dx, 0) + 3, y0 = by + max(dy, 0), y1 = by + min(dy, 0) + 3;
          if (!px) { x0 = max(x0, 0); x1 = min(x1, g.nx - 1); }
          if (!py) { y0 = max(y0, 0); y1 = min(y1, g.ny - 1); }
          near = x0 <= x1 && y0 <= y1;
        }
        const unsigned int hit = __ballot_sync(0xffffffffu, near);
        const int pos = nc + __popc(hit & ((1u << lane) - 1u));
        if (near && pos < kSliceRow) sh.cand[pos][l] = (unsigned short)m;
        nc += __popc(hit);
      }
      if (lane == 0) {
        sh.rows[l] = min(nc, kSliceRow);
        if (nc > kSliceRow) sh.bad = 1;
      }
    }
    __syncthreads();
    // their G_lm, a pair per thread, summed over the shared nodes in slot
    // order; rows padded to kRowHead with the marker itself at weight zero
#pragma unroll 1
    for (int q = mq; q < kSliceRow; q += mstep) {
      const int l = ml, c = sh.rows[l];
      if (q >= max(c, kRowHead)) break;
      int m = l;
      R acc = R(0);
      if (q < c) {
        m = sh.cand[q][l];
        const int dx = window_step(sh.bx[m] - sh.bx[l], g.nx, px), dy = window_step(sh.by[m] - sh.by[l], g.ny, py);
        bool has = false;
#pragma unroll 1
        for (int j = max(0, dy); j < min(4, 4 + dy); ++j)
#pragma unroll 1
          for (int i = max(0, dx); i < min(4, 4 + dx); ++i) {
            if (sh.at[4 * j + i][l] == 0xffff) continue;
            const R v = sh.w[4 * j + i][l] * sh.wds[4 * (j - dy) + i - dx][m];
            if (has) acc += v;
            else acc = v;
            has = true;
          }
      }
      sl.rw[(size_t)q * kSliceMarkers + l] = acc;
      sl.ri[(size_t)q * kSliceMarkers + l] = (unsigned short)m;
    }
    if (t < M) sl.rn[t] = sh.rows[t];
#pragma unroll 1
    for (int q = mq; q < kStencil; q += mstep) sl.w[(size_t)q * kSliceMarkers + ml] = sh.w[q][ml];
#pragma unroll 1
    for (int q = mq; q < kStencil / 2; q += mstep) {
      const unsigned int lo = sh.at[2 * q][ml], hi = sh.at[2 * q + 1][ml];
      sl.wi[(size_t)q * kSliceMarkers + ml] = (lo == 0xffff ? 0u : lo) | ((hi == 0xffff ? 0u : hi) << 16);
    }
    if (t < M) sl.mid[t] = t;
    for (int k = t; k < kSliceHead; k += NT) sl.head[k] = k < 3 ? nn : (k == 3 ? 0 : M);
  }
  __syncthreads();
  if (!sh.bad) {
    if (t == 0) { a.ctr[CTR_NBAND] = nn; a.ctr[CTR_NSEG] = min(sh.nseg, a.segcap); }
    return;
  }
  // the general path, by this CTA (what the list pass above has entered in the
  // maps leaves them first)
  for (int k = t; k < nn; k += NT) {
    const int n = sh.node[k], y = n / g.nx;
    a.node2band[n] = -1;
    a.segflag[y * a.nseg_x + (n - y * g.nx) / kSegW] = 0;
  }
  if (t == 0) sl.head[3] = 1;
  __syncthreads();
  const int T = M * kStencil;
  for (int k = t; k < T; k += NT)
    band_claim_item<R>(g, a.X, a.Y, a.W, a.node_of, a.node2band, a.claim, a.points, k);
  __syncthreads();
  for (int k = t; k < T; k += NT)
    band_alloc_item(a.node_of, a.claim, a.node2band, a.bnode, a.bcnt, a.ctr, a.bcap, k);
  __syncthreads();
  for (int k = t; k < T; k += NT)
    band_fill_item<R>(a.node_of, a.W, a.ds, a.node2band, a.band_of, a.bcnt, a.ent, a.ctr, k);
  __syncthreads();
  const int nnew = min(a.ctr[CTR_NBAND], a.bcap);
  for (int b = t; b < nnew; b += NT) band_sort_item<R>(a.bcnt, a.ent, b);
  for (int b = t; b < nnew; b += NT)
    band_segment_item(g, a.bnode, a.segflag, a.seglist, a.ctr, a.nseg_x, a.segcap, b);
  __syncthreads();
  for (int l = t; l < M; l += NT) build_g_item<R>(a.band_of, a.W, a.bcnt, a.ent, a.G, a.gcnt, a.ctr, l);
}

// ------------------------------------------------------------------ launchers
template <class R>
static SliceArgs<R> slice_args(const Ctx& h) {
  SliceArgs<R> s{};
  s.count = h.sl_count;
  s.S = h.sl_S;
  s.xmax = h.sl_xmax;
  s.x1max = h.sl_x1max;
  s.lmax = h.sl_lmax;
  s.emax = h.sl_emax;
  slice_bytes<R>(h.sl_count, (unsigned char*)h.sl_mem, &s);
  return s;
}

template <class R>
static cudaError_t rebuild_t(const Ctx& h, bool move, cudaStream_t s) {
  RebuildArgs<R> a{};
  a.g = h.geom;
  a.M = h.nm;
  a.nb = h.nb;
  a.points = h.desc.delta_points;
  a.nseg_x = h.nseg_x;
  a.bcap = h.bcap;
  a.segcap = h.segcap;
  a.move = move ? 1 : 0;
  a.xcap = h.sl_xmax;
  a.ecap = h.sl_emax;
  a.bodies = h.dbodies;
  a.mbody = h.dmbody;
  a.dX = h.ddX;
  a.dY = h.ddY;
  a.ds = h.dds;
  a.X = h.dX;
  a.Y = h.dY;
  a.Ux = (R*)h.dUx;
  a.Uy = (R*)h.dUy;
  a.node2band = h.dnode2band;
  a.bnode = h.dbnode;
  a.segflag = h.dsegflag;
  a.seglist = h.dseglist;
  a.ctr = h.dctr;
  a.W = (R*)h.dW;
  a.node_of = h.dnode_of;
  a.claim = h.dclaim;
  a.band_of = h.dband_of;
  a.bcnt = h.dbcnt;
  a.gcnt = h.dgcnt;
  a.ent = (Ent<R>*)h.dent;
  a.G = (Ent<R>*)h.dG;
  k_rebuild<R><<<1, kRebuildThreads, sizeof(RebuildShared<R>), s>>>(a, slice_args<R>(h));
  return cudaPeekAtLastError();
}

cudaError_t launch_rebuild(const Ctx& h, bool move, cudaStream_t s) {
  return h.r_bytes == 8 ? rebuild_t<double>(h, move, s) : rebuild_t<float>(h, move, s);
}

cudaError_t slice_rebuild_fits(const Ctx& h, bool* fits, cudaStream_t s) {
  const int* head = h.r_bytes == 8 ? slice_args<double>(h).head : slice_args<float>(h).head;
  int flag = 0;
  cudaError_t e = cudaMemcpyAsync(&flag, head + 3, sizeof(flag), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  *fits = e == cudaSuccess && flag == 0;
  return e;
}

template <class R>
static bool moving_fits_t(Ctx& h) {
  h.sl_count = 1;
  h.sl_S = h.nm;
  h.sl_lmax = (h.nm + 31) / 32 * 32;
  // a marker one lattice unit or less from the one before adds at most seven
  // nodes to its window's sixteen
  h.sl_xmax = h.sl_x1max = std::min(kSliceX1, (7 * h.nm + 32 + 31) / 32 * 32);
  h.sl_nseg = std::min(h.segcap, std::max(64, h.nm));
  if (cudaFuncSetAttribute(k_rebuild<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(RebuildShared<R>)) !=
      cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  for (int e : {12, 10, 8}) {
    h.sl_emax = e;
    if (slice_smem(h) > 0) return true;
  }
  return false;
}

bool slice_moving_fits(Ctx& h) {
  if (h.nm > kSliceMarkers || h.nb > kRebuildThreads) return false;
  return h.r_bytes == 8 ? moving_fits_t<double>(h) : moving_fits_t<float>(h);
}

int slice_max_corr() { return kSliceMaxCorr; }

size_t slice_mem_bytes(int prec, int count) {
  return prec == PREC_FP64 ? slice_bytes<double>(count, nullptr, nullptr)
                           : slice_bytes<float>(count, nullptr, nullptr);
}

template <class R>
static cudaError_t slice_build_t(const Ctx& h, int* stat, cudaStream_t s) {
  SliceArgs<R> a = slice_args<R>(h);
  cudaError_t e = cudaMemsetAsync(a.fin, 0, 2 * sizeof(int), s);
  if (e != cudaSuccess) return e;
  k_slice_build<R><<<h.sl_count, kSliceThreads, 0, s>>>(a, h.nm, h.desc.n_corr, h.dctr, h.dband_of, (const R*)h.dW,
                                                        h.dbnode, h.dbcnt, (const Ent<R>*)h.dent,
                                                        (const Ent<R>*)h.dG, h.dgcnt, stat);
  return cudaGetLastError();
}

cudaError_t launch_slice_build(const Ctx& h, int* stat, cudaStream_t s) {
  return h.r_bytes == 8 ? slice_build_t<double>(h, stat, s) : slice_build_t<float>(h, stat, s);
}

// Share of an SM's memory that both kernels of a step ask for as shared memory
// (100 KB), so that their blocks can be resident together: the correction
// takes 45 to 95 KB, and with each kernel's own choice of the split the 4096^2
// FP32 step took 206 us instead of 200 (at 72 % and more the loss of L1 cost
// as much).
constexpr int kStepCarveout = 44;

// Shared memory of the slice kernel for the planned slices, or 0 when the
// device cannot give it.
template <int P>
static size_t slice_smem_t(const Ctx& h) {
  const size_t need = slice_smem_bytes<typename Prec<P>::R>(h.sl_xmax, h.sl_x1max, h.sl_lmax, h.sl_emax, h.sl_S,
                                                            h.desc.n_corr, !h.any_moving);
  constexpr size_t kMax = 200 * 1024;
  if (need > kMax) return 0;
  bool ok = true;
  auto set = [&](auto kern, bool slice) {
    if (slice) ok = ok && cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMax) == cudaSuccess;
    ok = ok && cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, kStepCarveout) == cudaSuccess;
  };
  if (h.any_moving) {
    set(k_ib_slice<P, 0, true>, true);
    set(k_ib_slice<P, 1, true>, true);
  } else {
    set(k_ib_slice<P, 0, false>, true);
    set(k_ib_slice<P, 1, false>, true);
  }
  if (h.desc.collision == IBM_COLL_MRT) {
    set(k_slice_stream<P, 0, false, true>, false);
    set(k_slice_stream<P, 0, true, true>, false);
    set(k_slice_stream<P, 1, false, true>, false);
    set(k_slice_stream<P, 1, true, true>, false);
  } else {
    set(k_slice_stream<P, 0, false, false>, false);
    set(k_slice_stream<P, 0, true, false>, false);
    set(k_slice_stream<P, 1, false, false>, false);
    set(k_slice_stream<P, 1, true, false>, false);
  }
  if (!ok) {
    cudaGetLastError();
    return 0;
  }
  return need;
}

size_t slice_smem(const Ctx& h) {
  switch (h.prec) {
    case PREC_FP64: return slice_smem_t<PREC_FP64>(h);
    case PREC_FP32: return slice_smem_t<PREC_FP32>(h);
    case PREC_FP16_DEV: return slice_smem_t<PREC_FP16_DEV>(h);
    default: return slice_smem_t<PREC_BF16_DEV>(h);
  }
}

template <int P>
static void launch_slices(const Ctx& h, int parity, cudaStream_t s, const IbArgs<P>& a,
                          const SliceArgs<typename Prec<P>::R>& sl) {
  typedef typename Prec<P>::R R;
  const size_t smem = slice_smem_bytes<R>(sl.xmax, sl.x1max, sl.lmax, sl.emax, sl.S, a.N, !h.any_moving);
  const dim3 grid(sl.count), block(kSliceThreads);
  auto go = [&](auto kern) { launch_prio_smem(kern, grid, block, smem, s, h.ib_prio, a, sl); };
  if (h.any_moving) {
    if (parity == 0) go(k_ib_slice<P, 0, true>);
    else go(k_ib_slice<P, 1, true>);
  } else {
    if (parity == 0) go(k_ib_slice<P, 0, false>);
    else go(k_ib_slice<P, 1, false>);
  }
}

template <int P>
static void slice_loop_t(const Ctx& h, int parity, bool macro, cudaStream_t s) {
  typedef typename Prec<P>::R R;
  IbArgs<P> a = make_ib_args<P>(h);
  SliceArgs<R> sl = slice_args<R>(h);
  launch_slices<P>(h, parity, s, a, sl);
  const int nchunk = (h.nm + kForceChunk - 1) / kForceChunk;
  const dim3 g2(1 + nchunk + std::max(1, std::min(h.sl_nseg, 16 * h.ib_grid_max))), b2(kFinishThreads);
  auto go = [&](auto kern) { launch_prio(kern, g2, b2, s, h.ib_prio, a, sl); };
  if (a.c.mrt) {
    if (parity == 0) { if (macro) go(k_band_finish<P, 0, true, true>); else go(k_band_finish<P, 0, false, true>); }
    else { if (macro) go(k_band_finish<P, 1, true, true>); else go(k_band_finish<P, 1, false, true>); }
  } else {
    if (parity == 0) { if (macro) go(k_band_finish<P, 0, true, false>); else go(k_band_finish<P, 0, false, false>); }
    else { if (macro) go(k_band_finish<P, 1, true, false>); else go(k_band_finish<P, 1, false, false>); }
  }
}

// Grid of k_slice_stream; bx = 0 when it does not fit a launch.
template <int P, int PAR>
static StepShape step_shape(const Ctx& h, bool fprev, bool fnow) {
  constexpr int VEC = PAR ? VecTraits<P>::VEC_ODD : VecTraits<P>::VEC;
  const Geom& g = h.geom;
  StepShape sh;
  sh.bx = ((g.nx + 32 * VEC - 1) / (32 * VEC) + kStepThreads / 32 - 1) / (kStepThreads / 32);
  const long long per_row = (long long)sh.bx * kStepThreads;
  const long long edge = PAR ? edge_nodes(g, odd_edge<VEC>(g)) : 0;
  sh.edge_rows = (int)((edge + per_row - 1) / per_row);
  sh.span_rows = g.ny;
  sh.open = has_nee(g) ? (2 * g.ny + kStepThreads - 1) / kStepThreads : 0;
  const int nfin = 1 + (h.nm + kForceChunk - 1) / kForceChunk;
  sh.fprev = fprev ? nfin : 0;
  sh.fnow = fnow ? nfin : 0;
  // a segment per block while that fills the SMs, then one per warp
  sh.nblk = std::max({1, std::min(h.sl_nseg, 16 * h.ib_grid_max), (h.sl_nseg + kStepThreads / 32 - 1) / (kStepThreads / 32)});
  sh.head_rows = g.ny - g.ny / 4;
  sh.tail_rows = (int)(((long long)sh.open + sh.fprev + sh.fnow + sh.nblk + sh.bx - 1) / sh.bx);
  return sh;
}
static long long step_rows(const StepShape& sh) { return (long long)sh.edge_rows + sh.span_rows + sh.tail_rows; }

// The same answer for every step of the lattice.
template <int P>
static bool step_fits_t(const Ctx& h) { return step_rows(step_shape<P, 1>(h, true, true)) <= 65535; }
bool slice_step_fits(const Ctx& h) {
  switch (h.prec) {
    case PREC_FP64: return step_fits_t<PREC_FP64>(h);
    case PREC_FP32: return step_fits_t<PREC_FP32>(h);
    case PREC_FP16_DEV: return step_fits_t<PREC_FP16_DEV>(h);
    default: return step_fits_t<PREC_BF16_DEV>(h);
  }
}

template <int P, int PAR, bool MACRO, bool MRT>
static void launch_stream(const Ctx& h, cudaStream_t s, const IbArgs<P>& a,
                          const SliceArgs<typename Prec<P>::R>& sl, bool fprev, bool fnow) {
  const StepShape sh = step_shape<P, PAR>(h, fprev, fnow);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(sh.bx, (unsigned)step_rows(sh));
  cfg.blockDim = dim3(kStepThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_slice_stream<P, PAR, MACRO, MRT>, a, sl, (const int*)h.dsegflag, sh);
}

template <int P>
static bool slice_step_t(const Ctx& h, int parity, bool macro, bool fprev, bool fnow, cudaStream_t s) {
  if (!step_fits_t<P>(h)) return false;
  IbArgs<P> a = make_ib_args<P>(h);
  SliceArgs<typename Prec<P>::R> sl = slice_args<typename Prec<P>::R>(h);
  launch_slices<P>(h, parity, s, a, sl);
  if (a.c.mrt) {
    if (parity == 0) { if (macro) launch_stream<P, 0, true, true>(h, s, a, sl, fprev, fnow); else launch_stream<P, 0, false, true>(h, s, a, sl, fprev, fnow); }
    else { if (macro) launch_stream<P, 1, true, true>(h, s, a, sl, fprev, fnow); else launch_stream<P, 1, false, true>(h, s, a, sl, fprev, fnow); }
  } else {
    if (parity == 0) { if (macro) launch_stream<P, 0, true, false>(h, s, a, sl, fprev, fnow); else launch_stream<P, 0, false, false>(h, s, a, sl, fprev, fnow); }
    else { if (macro) launch_stream<P, 1, true, false>(h, s, a, sl, fprev, fnow); else launch_stream<P, 1, false, false>(h, s, a, sl, fprev, fnow); }
  }
  return true;
}

bool launch_slice_step(const Ctx& h, int parity, bool macro, bool fprev, bool fnow, cudaStream_t s) {
  if (!h.sl_on) return false;
  switch (h.prec) {
    case PREC_FP64: return slice_step_t<PREC_FP64>(h, parity, macro, fprev, fnow, s);
    case PREC_FP32: return slice_step_t<PREC_FP32>(h, parity, macro, fprev, fnow, s);
    case PREC_FP16_DEV: return slice_step_t<PREC_FP16_DEV>(h, parity, macro, fprev, fnow, s);
    default: return slice_step_t<PREC_BF16_DEV>(h, parity, macro, fprev, fnow, s);
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
