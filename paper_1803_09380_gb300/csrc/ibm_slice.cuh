// ibm_slice.cuh -- the correction loop of a step without any barrier between
// CTAs (arXiv 1803.09380, Eqs. 22-29), for boundaries whose markers keep
// their places.
//
// The Jacobi iteration couples a marker only with the markers whose supports
// share a node with its own (G_lm != 0): on a ring with markers one lattice
// unit apart, four or five to either side.  So the N iterations of a slice of
// S markers depend on nothing beyond N such hops, and one CTA can run the
// whole loop for its slice -- gather, interpolation, N iterations, the
// second moments, the summed correction of the nodes it owns -- from the
// uncorrected state alone, in shared memory, by also iterating the markers
// of that neighbourhood (depth 1 .. N around the slice).  The iterate A^n is
// only needed, and only computed, up to depth N - n + 1.  Nothing is written
// that another CTA reads, so there is no grid barrier and no need for the
// CTAs to be resident together; every element is formed by the arithmetic of
// ib_step_body in the same order, so the results are bitwise the same
// whatever the slices.
//
// Measured against the persistent kernel with its band collide (us per step,
// whole steps): 300^2 FP32 with 1029 markers 68.1 -> 12.0, 1024^2 FP32 with
// 3513 markers 72.3 -> 17.5, 4096^2 FP32 with 14052 markers beside
// collide+stream 220.8 -> 197.0, 64^2 FP64 with 220 markers 204.1 -> 35.8.
//
// What bounds it: latency.  The persistent kernel paid thirteen grid
// barriers, each followed by dependent loads from L2; here the only global
// round trips are the slice's lists and the gather, and an iteration is ten
// shared-memory loads and a block barrier.  The covering lists come to
// shared memory by asynchronous copies behind the iterations, and the
// residuals (a square root and a division each) are formed after the last
// iteration, for all iterations at once.  In FP64, whose arithmetic issues
// at two lanes a clock on an SM, work is dealt out so that whole warps are
// filled: (node, iteration) pairs in the second moments.  Loops are kept
// rolled: code that runs once per launch costs more to fetch than to execute.
#pragma once

#include "ibm_ib.cuh"

namespace ibm {

constexpr int kSliceThreads = 256;
constexpr int kSliceNodes = 2048;        // local band nodes
constexpr int kSliceX1 = 1280;           // local nodes whose second moments are formed
constexpr int kSliceRow = 32;            // coupled markers of one marker
constexpr int kSliceEnt = 16;            // covering markers of one node
constexpr int kSliceMaxCorr = 60;        // iterations
constexpr int kSliceHead = 4 + kSliceMaxCorr + 2;
constexpr int kSliceNodeHash = 4096, kSliceMarkHash = 1024;

// What the slices of a boundary hold, built once per band (k_slice_build).
// Lists are transposed (entry-major) so that a warp's loads are contiguous.
template <class R>
struct SliceArgs {
  int count, S;                // slices, owned markers of each
  int xmax, x1max;             // largest local node counts (shared-memory strides)
  int lmax, emax;              // largest marker count; most markers that cover a node
  int* head;                   // [count][kSliceHead]: owned nodes, nodes of depth <= 1
                               // markers, nodes, 0; then markers of depth <= h, h = 0 ..
  int* mid;                    // [count][kSliceMarkers] marker ids, by depth
  int* nid;                    // [count][kSliceNodes] lattice nodes: owned, depth <= 1, rest
  int* bid;                    // [count][kSliceX1] band index of the node
  R* w;                        // [count][kStencil][kSliceMarkers] stencil weights
  unsigned int* wi;            // [count][kStencil/2][kSliceMarkers] local nodes, two per word
  int* rn;                     // [count][kSliceMarkers] row lengths
  R* rw;                       // [count][kSliceRow][kSliceMarkers] G row weights
  unsigned short* ri;          // [count][kSliceRow][kSliceMarkers] local markers
  int* en;                     // [count][kSliceX1] covering markers of a node
  R* ew;                       // [count][kSliceEnt][kSliceX1] W_l ds_l
  unsigned short* ei;          // [count][kSliceEnt][kSliceX1] local markers
  R* rpart;                    // [2][count][kSliceMaxCorr + 2] the slices' residual maxima, by step parity
  int* fin;                    // [2] arrivals of the force chunks; zero between launches
};

// Device bytes of `count` slices, and the pieces of that block.
template <class R>
inline size_t slice_bytes(int count, unsigned char* base, SliceArgs<R>* s) {
  size_t used = 0;
  auto take = [&](size_t bytes) {
    unsigned char* p = base ? base + used : nullptr;
    used += (bytes + 255) & ~(size_t)255;
    return p;
  };
  const size_t n = (size_t)count;
  SliceArgs<R> t{};
  t.fin = (int*)take(2 * sizeof(int));
  t.head = (int*)take(n * kSliceHead * sizeof(int));
  t.mid = (int*)take(n * kSliceMarkers * sizeof(int));
  t.nid = (int*)take(n * kSliceNodes * sizeof(int));
  t.bid = (int*)take(n * kSliceX1 * sizeof(int));
  t.w = (R*)take(n * kStencil * kSliceMarkers * sizeof(R));
  t.wi = (unsigned int*)take(n * (kStencil / 2) * kSliceMarkers * sizeof(int));
  t.rn = (int*)take(n * kSliceMarkers * sizeof(int));
  t.rw = (R*)take(n * kSliceRow * kSliceMarkers * sizeof(R));
  t.ri = (unsigned short*)take(n * kSliceRow * kSliceMarkers * sizeof(short));
  t.en = (int*)take(n * kSliceX1 * sizeof(int));
  t.ew = (R*)take(n * kSliceEnt * kSliceX1 * sizeof(R));
  t.ei = (unsigned short*)take(n * kSliceEnt * kSliceX1 * sizeof(short));
  t.rpart = (R*)take(2 * n * (kSliceMaxCorr + 2) * sizeof(R));
  if (s) {
    t.count = s->count; t.S = s->S; t.xmax = s->xmax; t.x1max = s->x1max;
    t.lmax = s->lmax; t.emax = s->emax;
    *s = t;
  }
  return used;
}

// Dynamic shared memory of one slice CTA, in the order of its pieces: the A
// history, the owned markers' dj^n, (FP64, pairs) j^n of the depth <= 1 markers'
// nodes; rho, j of the nodes; sum_n j^n j^n; C; W / rho; rho* of the owned
// markers; the covering lists' weights and counts, the band indices, the
// lists' markers; the nodes of W / rho.
template <class R>
__host__ __device__ constexpr size_t slice_smem_bytes(int xmax, int x1max, int lmax, int emax, int S, int N,
                                                       bool pairs) {
  return 2 * sizeof(R) * ((size_t)(N + 1) * (lmax + ((S + 3) & ~3)) + (sizeof(R) == 8 && pairs ? (size_t)(N + 1) * x1max : 0)) +
         sizeof(R) * ((size_t)3 * xmax + (size_t)3 * x1max + (size_t)3 * lmax + ((S + 3) & ~3)) +
         (size_t)emax * x1max * (sizeof(R) + sizeof(short)) + (size_t)x1max * 2 * sizeof(int) +
         (size_t)kStencil * lmax * (sizeof(R) + sizeof(short));
}

}  // namespace ibm
