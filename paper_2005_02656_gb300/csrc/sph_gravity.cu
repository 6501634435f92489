// Self-gravity (sph_gravity in include/sph.h): section 4.1 evaluates it by a
// multipolar expansion on the tree used to find neighbours.  Here the tree's
// leaves are the occupied cells of the neighbour grid (side >= 2 h_max, in
// Morton order after the library's sort) and a node of level l groups the
// cells that share the top 3 l bits of their Morton code.
//
//   build     leaves from the occupied-cell list; each upper level by a flag
//             per run of equal parent codes (code >> 3) and an exclusive scan;
//             the levels above 4,096 nodes by one block
//   moments   leaves from their particles (mass, centre of mass c, traceless
//             quadrupole Q_ij = sum m (3 d_i d_j - |d|^2 delta_ij), d = x - c,
//             two passes); parents from their children by the parallel-axis
//             rule Q = sum (Q_k + M_k (3 e e^T - |e|^2 I)), e = c_k - c
//   walk      a node whose box does not contain the particle and whose longest
//             side s satisfies s < theta |x - c| adds the softened monopole and
//             the quadrupole term; an opened leaf adds its particles by the
//             direct softened formula; other nodes are opened.  A warp walks a
//             few consecutive particles together on one stack of (node, mask)
//             entries (k_walk, k_walk32).
// The tree is FP64, and both walks make the interactions of the oracle's
// recursion.
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include "sph_device.cuh"
#include "sph_internal.cuh"
#include "sph_scan.cuh"
#include "sph_walk.cuh"

namespace sph {
namespace grav {

struct Node {
  double box_lo[3], box_hi[3];
  double size, M;
  double c[3];
  double Q[6];      // xx xy xz yy yz zz
  int32_t first;    // first child (node index), -1 for a leaf
  int32_t nchild;
  int32_t p0, np;   // particles [p0, p0 + np) of the sorted order
};

constexpr int kStack = 80;  // >= 7 * 8 + 8 pending nodes for up to 8 Morton bits

__device__ __forceinline__ uint32_t compact3(uint32_t v) {
  uint32_t r = 0;
  for (int i = 0; i < 10; ++i) r |= ((v >> (3 * i)) & 1u) << i;
  return r;
}

// Box and longest side of the node with Morton prefix `code` at level `l`.
__device__ __forceinline__ void node_box(const Grid& g, uint32_t code, int l, Node& nd) {
  const int span = 1 << (g.bits - l);
  const uint32_t c3[3] = {compact3(code), compact3(code >> 1), compact3(code >> 2)};
  double size = 0.0;
  for (int ax = 0; ax < 3; ++ax) {
    const int c0 = (int)c3[ax] * span;
    int c1 = c0 + span - 1;
    if (c1 > g.nc[ax] - 1) c1 = g.nc[ax] - 1;
    nd.box_lo[ax] = g.lo[ax] + c0 * g.cs[ax];
    nd.box_hi[ax] = g.lo[ax] + (c1 + 1) * g.cs[ax];
    const double ext = nd.box_hi[ax] - nd.box_lo[ax];
    size = ext > size ? ext : size;
  }
  nd.size = size;
}

__global__ void k_leaves(const Grid* gp, const uint32_t* occ, const uint32_t* tbl_start,
                         const uint32_t* tbl_count, int64_t n_occ, uint32_t* code, Node* nodes,
                         StateView s) {
  const Grid g = *gp;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n_occ;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t cc = occ[i];
    code[i] = cc;
    Node nd;
    nd.first = -1;
    nd.nchild = 0;
    nd.p0 = (int32_t)tbl_start[cc];
    nd.np = (int32_t)tbl_count[cc];
    node_box(g, cc, g.bits, nd);
    double M = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
    for (int32_t b = nd.p0; b < nd.p0 + nd.np; ++b) {
      M += s.m[b];
      sx += s.m[b] * s.x[b];
      sy += s.m[b] * s.y[b];
      sz += s.m[b] * s.z[b];
    }
    nd.M = M;
    nd.c[0] = sx / M;
    nd.c[1] = sy / M;
    nd.c[2] = sz / M;
    double Q[6] = {0, 0, 0, 0, 0, 0};
    for (int32_t b = nd.p0; b < nd.p0 + nd.np; ++b) {
      const double dx = s.x[b] - nd.c[0], dy = s.y[b] - nd.c[1], dz = s.z[b] - nd.c[2];
      const double d2 = (dx * dx + dy * dy) + dz * dz;
      const double mb = s.m[b];
      Q[0] += mb * (3 * dx * dx - d2);
      Q[1] += mb * (3 * dx * dy);
      Q[2] += mb * (3 * dx * dz);
      Q[3] += mb * (3 * dy * dy - d2);
      Q[4] += mb * (3 * dy * dz);
      Q[5] += mb * (3 * dz * dz - d2);
    }
    for (int q = 0; q < 6; ++q) nd.Q[q] = Q[q];
    nodes[i] = nd;
  }
}

__global__ void k_run_flags(const uint32_t* code, int64_t m, int32_t* flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x)
    flag[i] = (i == 0 || (code[i] >> 3) != (code[i - 1] >> 3)) ? 1 : 0;
}

// Parents of the m children at nodes[coff ..): code, first child, first particle.
__global__ void k_parents(const uint32_t* code, const int32_t* flag, const int64_t* idx, int64_t m,
                          int64_t coff, int64_t poff, uint32_t* pcode, Node* nodes) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < m;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (!flag[i]) continue;
    const int64_t j = idx[i];
    pcode[j] = code[i] >> 3;
    nodes[poff + j].first = (int32_t)(coff + i);
    nodes[poff + j].p0 = nodes[coff + i].p0;
  }
}

// Child counts, particle counts, boxes and moments (parallel-axis rule).
__device__ __forceinline__ void parent_moments(const Grid& g, const uint32_t* pcode, int64_t npar,
                                               int64_t m, int64_t coff, int64_t poff, int level,
                                               Node* nodes, int64_t j0, int64_t stride) {
  for (int64_t j = j0; j < npar; j += stride) {
    Node nd = nodes[poff + j];
    const int64_t f = nd.first - coff;
    const int64_t next = j + 1 < npar ? nodes[poff + j + 1].first - coff : m;
    nd.nchild = (int32_t)(next - f);
    const Node& last = nodes[coff + next - 1];
    nd.np = last.p0 + last.np - nd.p0;
    node_box(g, pcode[j], level, nd);
    double M = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
    for (int64_t k = coff + f; k < coff + next; ++k) {
      const Node& ch = nodes[k];
      M += ch.M;
      sx += ch.M * ch.c[0];
      sy += ch.M * ch.c[1];
      sz += ch.M * ch.c[2];
    }
    nd.M = M;
    nd.c[0] = sx / M;
    nd.c[1] = sy / M;
    nd.c[2] = sz / M;
    double Q[6] = {0, 0, 0, 0, 0, 0};
    for (int64_t k = coff + f; k < coff + next; ++k) {
      const Node& ch = nodes[k];
      const double ex = ch.c[0] - nd.c[0], ey = ch.c[1] - nd.c[1], ez = ch.c[2] - nd.c[2];
      const double e2 = (ex * ex + ey * ey) + ez * ez;
      Q[0] += ch.Q[0] + ch.M * (3 * ex * ex - e2);
      Q[1] += ch.Q[1] + ch.M * (3 * ex * ey);
      Q[2] += ch.Q[2] + ch.M * (3 * ex * ez);
      Q[3] += ch.Q[3] + ch.M * (3 * ey * ey - e2);
      Q[4] += ch.Q[4] + ch.M * (3 * ey * ez);
      Q[5] += ch.Q[5] + ch.M * (3 * ez * ez - e2);
    }
    for (int q = 0; q < 6; ++q) nd.Q[q] = Q[q];
    nodes[poff + j] = nd;
  }
}

__global__ void k_parent_moments(const Grid* gp, const uint32_t* pcode, int64_t npar, int64_t m,
                                 int64_t coff, int64_t poff, int level, Node* nodes) {
  parent_moments(*gp, pcode, npar, m, coff, poff, level, nodes,
                 blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

// The levels above a level of m <= kTopNodes nodes, by one block: runs of equal
// parent codes, parents and moments as above, level after level, without the
// host's round trip per level (six launches and a copy back, some 35 us each: most
// of a small call).  *n_nodes receives the number of nodes; the root is the last.
constexpr int kTopThreads = 1024;
constexpr int kTopNodes = 4096;

__global__ void __launch_bounds__(kTopThreads) k_top(const Grid* gp, uint32_t* code,
                                                     uint32_t* pcode, int64_t m, int64_t coff,
                                                     int64_t noff, int level, Node* nodes,
                                                     int64_t* n_nodes) {
  constexpr int kEach = kTopNodes / kTopThreads;
  __shared__ int sh[32];
  const Grid& g = *gp;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  for (int l = level; l >= 0; --l) {
    // exclusive ranks of the runs' first children
    int flag[kEach], sum = 0;
#pragma unroll
    for (int q = 0; q < kEach; ++q) {
      const int i = kEach * tid + q;
      flag[q] = i < m && (i == 0 || (code[i] >> 3) != (code[i - 1] >> 3));
      sum += flag[q];
    }
    int incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) sh[w] = incl;
    __syncthreads();
    if (w == 0) {
      int t = sh[lane];
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, t, o);
        if (lane >= o) t += u;
      }
      sh[lane] = t;
    }
    __syncthreads();
    int j = incl - sum + (w > 0 ? sh[w - 1] : 0);
    const int npar = sh[31];
#pragma unroll
    for (int q = 0; q < kEach; ++q) {
      const int i = kEach * tid + q;
      if (flag[q]) {
        pcode[j] = code[i] >> 3;
        nodes[noff + j].first = (int32_t)(coff + i);
        nodes[noff + j].p0 = nodes[coff + i].p0;
        ++j;
      }
    }
    __syncthreads();
    parent_moments(g, pcode, npar, m, coff, noff, l, nodes, tid, kTopThreads);
    __syncthreads();
    uint32_t* t = code;
    code = pcode;
    pcode = t;
    coff = noff;
    noff += npar;
    m = npar;
  }
  if (tid == 0) *n_nodes = noff;
}

// The opening decision: accept a node whose box does not contain p and whose
// longest side is below theta |p - c| (r = p - c, R2, R returned).
__device__ __forceinline__ bool accept64(const Node& nd, const double p[3], double theta,
                                         double r[3], double& R2, double& R) {
  bool inside = true;
  for (int ax = 0; ax < 3; ++ax)
    if (p[ax] < nd.box_lo[ax] || p[ax] > nd.box_hi[ax]) inside = false;
  for (int ax = 0; ax < 3; ++ax) r[ax] = p[ax] - nd.c[ax];
  R2 = (r[0] * r[0] + r[1] * r[1]) + r[2] * r[2];
  R = sqrt(R2);
  return !inside && nd.size < theta * R;
}

constexpr int kWalkWarps = 4;

// ---- opening decisions in FP32 --------------------------------------------
// FP64 runs at 1/64 of the FP32 rate on this part, so both walks decide in
// FP32, exactly (accept_mixed), and the FP32-mixed one evaluates its terms in
// FP32 as well.  Coordinates are taken relative to the grid origin lo and split into
// an FP32 head and tail (v = hi + lo to about 2^-48 |v|), so r = x_a - c is
// (hi_a - hi_c) + (lo_a - lo_c) with FP32 rounding relative to |r| instead of
// to the box.  Each particle is stored relative to its leaf's centre of mass,
// so a lane that opens a leaf forms x_a - x_b as r - (x_b - c).

// 1 / sqrt(x), relative error below 2^-22, without the handling of subnormal x
// (coordinates are scaled to [0, 2), so x is subnormal only for coincident points)
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct NodeF {     // 96 B, read with uniform (broadcast) loads
  float4 cm;       // hi(c - lo), M
  float4 q1;       // Q yz zz, size, lo(c - lo).x
  float4 lo;       // box_lo - lo, lo(c - lo).y
  float4 hi;       // box_hi - lo, lo(c - lo).z
  float4 q0;       // Q xx xy xz yy
  int4 t;          // first, nchild, p0, np
};

__device__ __forceinline__ void split2(double v, float& hi, float& lo) {
  hi = (float)v;
  lo = (float)(v - (double)hi);
}

// FP32 records of the nodes, coordinates and sizes scaled by `sc` (a power of two).
__global__ void k_nodes32(const Node* nodes, const int64_t* n_nodes, double lx, double ly, double lz, double sc,
                          NodeF* out) {
  const double s2 = sc * sc;
  const int64_t nn = *n_nodes;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nn;
       k += (int64_t)gridDim.x * blockDim.x) {
    const Node& nd = nodes[k];
    float ch[3], cl[3];
    split2((nd.c[0] - lx) * sc, ch[0], cl[0]);
    split2((nd.c[1] - ly) * sc, ch[1], cl[1]);
    split2((nd.c[2] - lz) * sc, ch[2], cl[2]);
    NodeF f;
    f.cm = make_float4(ch[0], ch[1], ch[2], (float)nd.M);
    f.q1 = make_float4((float)(nd.Q[4] * s2), (float)(nd.Q[5] * s2), (float)(nd.size * sc), cl[0]);
    f.lo = make_float4((float)((nd.box_lo[0] - lx) * sc), (float)((nd.box_lo[1] - ly) * sc),
                       (float)((nd.box_lo[2] - lz) * sc), cl[1]);
    f.hi = make_float4((float)((nd.box_hi[0] - lx) * sc), (float)((nd.box_hi[1] - ly) * sc),
                       (float)((nd.box_hi[2] - lz) * sc), cl[2]);
    f.q0 = make_float4((float)(nd.Q[0] * s2), (float)(nd.Q[1] * s2), (float)(nd.Q[2] * s2),
                       (float)(nd.Q[3] * s2));
    f.t = make_int4(nd.first, nd.nchild, nd.p0, nd.np);
    out[k] = f;
  }
}

// The particles of leaf k relative to its centre of mass, in FP32 and by pairs
// (x0 x1 y0 y1), (z0 z1 m0 m1), so that two are taken per paired FP32 operation;
// an odd leaf's last pair ends with a massless particle far away.  Leaf k's
// pairs start at (p0 + k + 1) / 2, which leaves room for the odd ones before it.
__host__ __device__ __forceinline__ int64_t pair_base(int64_t p0, int64_t k) {
  return (p0 + k + 1) >> 1;
}
constexpr float kFarAway = 1.0e18f;

__global__ void k_leaf_pairs(const Node* nodes, int64_t n_leaves, StateView s, double sc,
                             float4* po) {
  // 16 lanes take a leaf, a lane a pair
  const int64_t groups = ((int64_t)gridDim.x * blockDim.x) >> 4;
  for (int64_t k = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 4; k < n_leaves;
       k += groups) {
    const Node& nd = nodes[k];
    const double cx = nd.c[0], cy = nd.c[1], cz = nd.c[2];
    const int64_t base = pair_base(nd.p0, k);
    for (int j = threadIdx.x & 15; 2 * j < nd.np; j += 16) {
      const int32_t b0 = nd.p0 + 2 * j, b1 = b0 + 1;
      const float x0 = f32_rn((s.x[b0] - cx) * sc), y0 = f32_rn((s.y[b0] - cy) * sc),
                  z0 = f32_rn((s.z[b0] - cz) * sc);
      float x1 = kFarAway, y1 = 0.f, z1 = 0.f, m1 = 0.f;
      if (2 * j + 1 < nd.np) {
        x1 = f32_rn((s.x[b1] - cx) * sc);
        y1 = f32_rn((s.y[b1] - cy) * sc);
        z1 = f32_rn((s.z[b1] - cz) * sc);
        m1 = f32_rn(s.m[b1]);
      }
      po[2 * (base + j)] = make_float4(x0, x1, y0, y1);
      po[2 * (base + j) + 1] = make_float4(z0, z1, f32_rn(s.m[b0]), m1);
    }
  }
}

// Constants of the FP32 walk, converted on the host.
struct Walk32Consts {
  double lx, ly, lz;   // grid origin
  double sc;           // scale of the FP32 coordinates, a power of two
  double theta;        // for the FP64 decision
  float eps2, th;      // eps^2 scaled, theta
  double Gs;           // G with the scale of the terms (sc^2)
  float mb;            // box-face margin: covers the FP32 rounding of box and head
  float aL;            // absolute distance margin
};

// Node k as a target at head ph and tail pl sees it.
struct NodeSeen {
  float4 cm, q1;
  int4 t;
  float r[3], R2, inv_R;
};

// The opening decision for one target, in FP32 with margins that cover the
// rounding of the stored box faces and of the particle's head (each <= L
// 2^-24, L the grid's largest extent) and of the FP32 distance (relative
// 2^-22 with rsqrtf): mb on a box face, aL + 2e-6 R on the distance.  Inside a
// margin, and wherever an FP32 value is not finite, the FP64 decision
// (accept64 on the FP64 node) is taken, so the nodes accepted and opened are
// exactly those of an FP64 walk.  `live`: false leaves the decision out.
__device__ __forceinline__ bool accept_mixed(const Node* nodes, const NodeF* nf, int32_t k,
                                             const float ph[3], const float pl[3], bool live,
                                             const StateView& s, int64_t a,
                                             const Walk32Consts& k32, NodeSeen& v) {
  const NodeF* f = nf + k;
  v.cm = __ldg(&f->cm);
  v.q1 = __ldg(&f->q1);
  const float4 blo = __ldg(&f->lo), bhi = __ldg(&f->hi);
  v.t = __ldg(&f->t);
  v.r[0] = (ph[0] - v.cm.x) + (pl[0] - v.q1.w);
  v.r[1] = (ph[1] - v.cm.y) + (pl[1] - blo.w);
  v.r[2] = (ph[2] - v.cm.z) + (pl[2] - bhi.w);
  bool accept = false;
  if (live) {
    v.R2 = fmaf(v.r[2], v.r[2], fmaf(v.r[1], v.r[1], v.r[0] * v.r[0]));
    v.inv_R = rsqrt_ftz(v.R2);
    const float Rf = v.R2 * v.inv_R;
    const float size = v.q1.z, mb = k32.mb;
    // the box: certainly outside, certainly inside, or within mb of a face.
    // dmin is the smallest signed distance of the particle to a face
    // (negative outside); its own rounding (<= L 2^-24) adds to the
    // stored faces' and the head's, all within mb = 4 L 2^-24.
    const float dmin =
        fminf(fminf(fminf(ph[0] - blo.x, bhi.x - ph[0]), fminf(ph[1] - blo.y, bhi.y - ph[1])),
              fminf(ph[2] - blo.z, bhi.z - ph[2]));
    const bool out_c = dmin < -mb;
    const bool in_c = dmin >= mb;
    const bool acc_c = size * (1.f + 1e-6f) < k32.th * (Rf * (1.f - 2e-6f) - k32.aL);
    const bool rej_c = size * (1.f - 1e-6f) > k32.th * (Rf * (1.f + 2e-6f) + k32.aL);
    if (in_c || rej_c) {
      accept = false;
    } else if (out_c && acc_c) {
      accept = true;
    } else {
      // FP64 positions are reloaded here rather than kept live across the walk
      const double p[3] = {s.x[a], s.y[a], s.z[a]};
      double r64[3], R2_64, R64;
      accept = accept64(nodes[k], p, k32.theta, r64, R2_64, R64);
    }
  }
  return accept;
}

// ---- FP64 walk ------------------------------------------------------------
// A warp walks kTile64 consecutive targets together on one stack, with the
// FP32 decisions of accept_mixed, and only queues what it accepts: per lane one
// ring of accepted nodes and one of opened leaves in shared memory.  kLanes64
// lanes share a target: they take the same decisions, and every kLanes64-th of
// its node terms and leaf particles each, added at the end by a fixed butterfly.
// The FP64 terms are evaluated from the rings, each lane taking its own next
// term, so the FP64 pipe (which bounds the kernel, at 2 operations per clock
// and SM; 87% busy) works on full warps: a warp that evaluates a term where it
// meets it has 18 of its 32 lanes in it, because lanes that did not open the
// parent or that open the node itself sit it out.  FP64 operations per node
// term 42, per leaf particle 16 (G is applied once per target; inv_root).
// Uniform sphere, theta = 0.5, whole call: 137,376 particles 28.6 -> 10.4 ms,
// 2,176 particles 2.19 -> 0.63 ms (one lane per target and full rings: 12.5 and
// 1.62 ms; 4 lanes: 10.4 and 0.78 ms).
constexpr int kLanes64 = 8;
constexpr int kTile64 = 32 / kLanes64;
constexpr int kRing = 32;       // entries per lane and ring
constexpr int kDrainLanes = 28; // evaluate while at least so many lanes hold a term

__global__ void __launch_bounds__(32 * kWalkWarps) k_walk(const Node* nodes, const NodeF* nf,
                                                          const int64_t* n_nodes, StateView s,
                                                          int64_t n, Walk32Consts k32, double G,
                                                          double eps2,
                                                          double* gx, double* gy, double* gz,
                                                          unsigned long long* stats,
                                                          uint32_t* err) {
  __shared__ int32_t st_node[kWalkWarps][kStack];
  __shared__ uint32_t st_mask[kWalkWarps][kStack];
  __shared__ int32_t ring_node[kWalkWarps][kRing][32];
  __shared__ int32_t ring_leaf[kWalkWarps][kRing][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int sub = lane % kLanes64;
  const int32_t root = (int32_t)(*n_nodes - 1);
  unsigned long long nodes_used = 0, pairs = 0;
  const int64_t tiles = (n + kTile64 - 1) / kTile64;
  for (int64_t tile = blockIdx.x * (int64_t)kWalkWarps + w; tile < tiles;
       tile += (int64_t)gridDim.x * kWalkWarps) {
    const int64_t a = tile * kTile64 + lane / kLanes64;
    const bool valid = a < n;
    const int32_t a32 = valid ? (int32_t)a : -1;
    const double p[3] = {valid ? s.x[a] : 0.0, valid ? s.y[a] : 0.0, valid ? s.z[a] : 0.0};
    float ph[3], pl[3];
    split2((p[0] - k32.lx) * k32.sc, ph[0], pl[0]);
    split2((p[1] - k32.ly) * k32.sc, ph[1], pl[1]);
    split2((p[2] - k32.lz) * k32.sc, ph[2], pl[2]);
    double acc[3] = {0.0, 0.0, 0.0};
    uint32_t accepted = 0;
    uint32_t n_in = 0, n_out = 0;      // ring positions: nodes queued and evaluated
    uint32_t l_in = 0, l_out = 0;      // leaves queued and begun
    int32_t cur = 0, end = 0;          // particles of the leaf under evaluation

    // Evaluates queued node terms (a term of every lane that has one per turn):
    // while at least `lanes` lanes take part, and `turns` turns in any case.
    auto drain_nodes = [&](int lanes, int turns) {
      for (;; --turns) {
        const bool have = n_out != n_in;
        const uint32_t m = __ballot_sync(0xffffffffu, have);
        if (m == 0 || (turns <= 0 && __popc(m) < lanes)) break;
        if (have) {
          const Node& nd = nodes[ring_node[w][n_out % kRing][lane]];
          ++n_out;
          const double r[3] = {p[0] - nd.c[0], p[1] - nd.c[1], p[2] - nd.c[2]};
          const double R2 = (r[0] * r[0] + r[1] * r[1]) + r[2] * r[2];
          const double inv_R = inv_root(R2);
          const double inv_s = eps2 > 0.0 ? inv_root(R2 + eps2) : inv_R;
          const double mono = nd.M * (inv_s * inv_s * inv_s);
          const double j2 = inv_R * inv_R;
          const double g5 = j2 * j2 * inv_R;
          const double* Q = nd.Q;
          const double Qr[3] = {Q[0] * r[0] + Q[1] * r[1] + Q[2] * r[2],
                                Q[1] * r[0] + Q[3] * r[1] + Q[4] * r[2],
                                Q[2] * r[0] + Q[4] * r[1] + Q[5] * r[2]};
          const double rQr = r[0] * Qr[0] + r[1] * Qr[1] + r[2] * Qr[2];
          const double kr = fma(-2.5, g5 * (rQr * j2), -mono);
          for (int i = 0; i < 3; ++i) acc[i] = fma(kr, r[i], fma(g5, Qr[i], acc[i]));
        }
      }
    };
    // The same for the particles of queued leaves, in order, the target left out.
    auto drain_leaves = [&](int lanes, uint32_t room) {
      for (;;) {
        if (cur == a32) cur += kLanes64;
        while (cur >= end && l_out != l_in) {
          const int4 t = __ldg(&nf[ring_leaf[w][l_out % kRing][lane]].t);
          ++l_out;
          cur = t.z + sub == a32 ? a32 + kLanes64 : t.z + sub;
          end = t.z + t.w;
        }
        const bool have = cur < end;
        const uint32_t m = __ballot_sync(0xffffffffu, have);
        const bool full = __any_sync(0xffffffffu, l_in - l_out > room);
        if (m == 0 || (!full && __popc(m) < lanes)) break;
        if (have) {
          const int32_t b = cur;
          cur += kLanes64;
          const double d[3] = {p[0] - s.x[b], p[1] - s.y[b], p[2] - s.z[b]};
          const double inv =
              inv_root(fma(d[2], d[2], fma(d[1], d[1], fma(d[0], d[0], eps2))));
          const double f = s.m[b] * (inv * inv * inv);
          for (int q = 0; q < 3; ++q) acc[q] = fma(-f, d[q], acc[q]);
          ++pairs;
        }
      }
    };

    int sp = 0;
    const uint32_t all = __ballot_sync(0xffffffffu, valid);
    if (lane == 0) {
      st_node[w][0] = root;
      st_mask[w][0] = all;
    }
    sp = 1;
    __syncwarp();
    bool overflow = false;
    while (sp > 0) {
      --sp;
      const int32_t k = st_node[w][sp];
      const uint32_t mask = st_mask[w][sp];
      __syncwarp();
      const bool live = (mask >> lane) & 1u;
      NodeSeen v;
      const bool accept = accept_mixed(nodes, nf, k, ph, pl, live, s, a, k32, v);
      const bool open = live && !accept;
      if (accept && (accepted++ % kLanes64 == (uint32_t)sub)) {
        ring_node[w][n_in % kRing][lane] = k;
        ++n_in;
        ++nodes_used;
      }
      const uint32_t omask = __ballot_sync(0xffffffffu, open);
      if (__any_sync(0xffffffffu, n_in - n_out == kRing)) drain_nodes(kDrainLanes, 1);
      if (omask == 0) continue;
      if (v.t.x < 0) {
        if (open) {
          ring_leaf[w][l_in % kRing][lane] = k;
          ++l_in;
        }
        if (__any_sync(0xffffffffu, l_in - l_out == kRing)) drain_leaves(kDrainLanes, kRing - 1);
      } else {
        if (sp + v.t.y > kStack) {  // cannot happen for <= 8 Morton bits; kept as a guard
          overflow = true;
          break;
        }
        if (lane == 0)
          for (int j = v.t.y - 1, q = sp; j >= 0; --j, ++q) {
            st_node[w][q] = v.t.x + j;
            st_mask[w][q] = omask;
          }
        sp += v.t.y;
        __syncwarp();
      }
    }
    drain_nodes(0, 0);
    drain_leaves(0, kRing);
    if (overflow && lane == 0) raise_flag(err, SPH_FLAG_CELL_OVERFLOW);
#pragma unroll
    for (int q = 0; q < 3; ++q)
#pragma unroll
      for (int o = kLanes64 / 2; o > 0; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
    if (valid && sub == 0) {
      gx[a] = G * acc[0];
      gy[a] = G * acc[1];
      gz[a] = G * acc[2];
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    nodes_used += __shfl_xor_sync(0xffffffffu, nodes_used, o);
    pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
  }
  if (lane == 0) {
    atomicAdd(stats, nodes_used);
    atomicAdd(stats + 1, pairs);
  }
}

// ---- FP32-mixed walk ------------------------------------------------------
// A warp walks kTile32 consecutive sorted targets on one stack of (node, mask of
// the targets that reached it through nodes they opened).  It pops up to 32
// nodes at a time and tests each against the bounding box of all its targets,
// one node per lane: most nodes are certainly accepted or certainly opened by
// every target in the box, with the margins of accept_mixed, so that one lane's
// test stands for all.  The nodes that the box cannot decide take each target's
// own decision (accept_mixed), so every target makes exactly the interactions of
// a walk of its own.  Two lanes share a target: accepted nodes, undecided nodes
// and the particle pairs of opened leaves go to them in turn (a load is then two
// broadcasts).  16 targets lie closer together than 32, so fewer nodes stay
// undecided and fewer leaves are opened for some targets only: 1,660 leaf
// particles per tile against 2,100, of which a target needs 730.
// Instruction issue (71% of cycles) and the L1 data pipe (67%) bound the kernel.
// 998,317 particles, theta = 0.5: walk 7.10 -> 4.67 ms with 8 CTAs per SM (64 registers;
// 6 CTAs: 5.1 ms); whole call 7.95 -> 5.29 ms (32 targets, scalar particles: 6.31 ms),
// 17,256 particles 1.15 -> 0.48 ms.
constexpr int kTile32 = 16;

struct Walk32Smem {
  int2 st[kStack32];   // nodes to visit
  int2 acc[32];        // of one turn: accepted by all lanes of their mask
  int2 mix[32];        //   to be decided per lane
  int2 leaf[32];       //   opened leaves
};

__device__ __forceinline__ float2 f2(float v) { return make_float2(v, v); }

__global__ void __launch_bounds__(32 * kWalkWarps, 8) k_walk32(const Node* nodes,
                                                            const NodeF* nf, const float4* po,
                                                            const int64_t* n_nodes, StateView s,
                                                            int64_t n, Walk32Consts k32,
                                                            double* gx, double* gy, double* gz,
                                                            unsigned long long* stats,
                                                            uint32_t* err) {
  __shared__ Walk32Smem smem[kWalkWarps];
  const int lane = threadIdx.x & 31, tl = lane % kTile32, half = lane / kTile32;
  Walk32Smem& W = smem[threadIdx.x >> 5];
  const uint32_t lt = (1u << lane) - 1u;
  const int32_t root = (int32_t)(*n_nodes - 1);
  unsigned long long nodes_used = 0, pairs = 0;
  const int64_t tiles = (n + kTile32 - 1) / kTile32;
  for (int64_t tile = blockIdx.x * (int64_t)kWalkWarps + (threadIdx.x >> 5); tile < tiles;
       tile += (int64_t)gridDim.x * kWalkWarps) {
    const int64_t a = tile * kTile32 + tl;
    const bool valid = a < n;
    const int32_t a32 = valid ? (int32_t)a : -1;
    float ph[3], pl[3];
    split2(((valid ? s.x[a] : 0.0) - k32.lx) * k32.sc, ph[0], pl[0]);
    split2(((valid ? s.y[a] : 0.0) - k32.ly) * k32.sc, ph[1], pl[1]);
    split2(((valid ? s.z[a] : 0.0) - k32.lz) * k32.sc, ph[2], pl[2]);
    // the targets' box (heads); a NaN or infinite coordinate decides nothing
    float glo[3], ghi[3];
    bool fine = true;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      fine = fine && isfinite(ph[ax]);
      glo[ax] = valid ? ph[ax] : INFINITY;
      ghi[ax] = valid ? ph[ax] : -INFINITY;
#pragma unroll
      for (int o = kTile32 / 2; o > 0; o >>= 1) {
        glo[ax] = fminf(glo[ax], __shfl_xor_sync(0xffffffffu, glo[ax], o));
        ghi[ax] = fmaxf(ghi[ax], __shfl_xor_sync(0xffffffffu, ghi[ax], o));
      }
    }
    fine = __all_sync(0xffffffffu, fine);
    float acc[3] = {0.f, 0.f, 0.f};                       // node terms
    float2 px = f2(0.f), py = f2(0.f), pz = f2(0.f);      // particle terms, negative
    uint32_t used = 0, npair = 0;
    // the terms of an accepted node, without G
    auto node_terms = [&](const float r[3], float M, float4 q0, float q4, float q5, float R2,
                          float inv_R) {
      const float inv_s = rsqrt_ftz(R2 + k32.eps2);
      const float inv_R2 = inv_R * inv_R;
      const float g5 = inv_R2 * inv_R2 * inv_R;
      const float Qr[3] = {q0.x * r[0] + q0.y * r[1] + q0.z * r[2],
                           q0.y * r[0] + q0.w * r[1] + q4 * r[2],
                           q0.z * r[0] + q4 * r[1] + q5 * r[2]};
      const float rQr = r[0] * Qr[0] + r[1] * Qr[1] + r[2] * Qr[2];
      const float kr = -(M * (inv_s * inv_s * inv_s)) - 2.5f * g5 * rQr * inv_R2;
#pragma unroll
      for (int i = 0; i < 3; ++i) acc[i] = fmaf(kr, r[i], fmaf(g5, Qr[i], acc[i]));
    };
    const uint32_t all = __ballot_sync(0xffffffffu, valid) & 0xffffu;
    if (lane == 0) W.st[0] = make_int2(root, (int)all);
    int sp = 1;
    __syncwarp();
    while (walk_on(sp)) {
      const int take = walk_take(sp);
      const bool have = lane < take;
      const int2 e = have ? W.st[sp - 1 - lane] : make_int2(0, 0);
      sp -= take;
      __syncwarp();
      int cls = 0;  // 1 accepted, 2 opened, 3 per lane
      int4 t = make_int4(0, 0, 0, 0);
      if (have) {
        const NodeF* f = nf + e.x;
        const float4 cm = __ldg(&f->cm), blo = __ldg(&f->lo), bhi = __ldg(&f->hi);
        const float size = __ldg(&f->q1.z), mb = k32.mb;
        t = __ldg(&f->t);
        const float c[3] = {cm.x, cm.y, cm.z}, bl[3] = {blo.x, blo.y, blo.z},
                    bh[3] = {bhi.x, bhi.y, bhi.z};
        bool apart = false, inside = true;
        float mn2 = 0.f, mx2 = 0.f;
#pragma unroll
        for (int ax = 0; ax < 3; ++ax) {
          apart = apart || glo[ax] - bh[ax] > mb || bl[ax] - ghi[ax] > mb;
          inside = inside && glo[ax] - bl[ax] >= mb && bh[ax] - ghi[ax] >= mb;
          const float u = glo[ax] - c[ax], v = c[ax] - ghi[ax];
          const float dn = fmaxf(fmaxf(u, v), 0.f), dx = fmaxf(fabsf(u), fabsf(v));
          mn2 = fmaf(dn, dn, mn2);
          mx2 = fmaf(dx, dx, mx2);
        }
        // distances within aL + 2e-6 R of every lane's own (heads only: at most
        // 3 sqrt(3) L 2^-24 off)
        const float Rn = sqrtf(mn2), Rx = sqrtf(mx2);
        const bool near_ = size * (1.f + 1e-6f) < k32.th * (Rn * (1.f - 2e-6f) - k32.aL);
        const bool far_ = size * (1.f - 1e-6f) > k32.th * (Rx * (1.f + 2e-6f) + k32.aL);
        cls = !fine ? 3 : (inside || far_ ? 2 : (apart && near_ ? 1 : 3));
      }
      const uint32_t am = __ballot_sync(0xffffffffu, cls == 1);
      const uint32_t xm = __ballot_sync(0xffffffffu, cls == 3);
      const bool leaf = cls == 2 && t.x < 0;
      const uint32_t lm = __ballot_sync(0xffffffffu, leaf);
      if (cls == 1) W.acc[__popc(am & lt)] = e;
      if (cls == 3) W.mix[__popc(xm & lt)] = e;
      if (leaf) W.leaf[__popc(lm & lt)] = e;
      int nleaf = __popc(lm);
      // children of the opened nodes
      const int nch = cls == 2 && !leaf ? t.y : 0;
      int incl = nch;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int q = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += q;
      }
      for (int j = 0; j < nch; ++j) W.st[sp + incl - nch + j] = make_int2(t.x + j, e.y);
      sp += __shfl_sync(0xffffffffu, incl, 31);
      __syncwarp();
      const int na = __popc(am), nx = __popc(xm);
      for (int i = half; i < na; i += 2) {
        const int2 en = W.acc[i];
        const NodeF* f = nf + en.x;
        const float4 cm = __ldg(&f->cm), q1 = __ldg(&f->q1), q0 = __ldg(&f->q0);
        const float ly = __ldg(&f->lo.w), lz = __ldg(&f->hi.w);
        if (((uint32_t)en.y >> tl) & 1u) {
          const float r[3] = {(ph[0] - cm.x) + (pl[0] - q1.w), (ph[1] - cm.y) + (pl[1] - ly),
                              (ph[2] - cm.z) + (pl[2] - lz)};
          const float R2 = fmaf(r[2], r[2], fmaf(r[1], r[1], r[0] * r[0]));
          node_terms(r, cm.w, q0, q1.x, q1.y, R2, rsqrt_ftz(R2));
          ++used;
        }
      }
      for (int i = 0; i < nx; i += 2) {
        const int2 en = W.mix[min(i + half, nx - 1)];
        const bool live = i + half < nx && (((uint32_t)en.y >> tl) & 1u);
        NodeSeen v;
        const bool accept = accept_mixed(nodes, nf, en.x, ph, pl, live, s, a, k32, v);
        if (accept) {
          node_terms(v.r, v.cm.w, __ldg(&nf[en.x].q0), v.q1.x, v.q1.y, v.R2, v.inv_R);
          ++used;
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, live && !accept);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const uint32_t omask = (bal >> (16 * q)) & 0xffffu;
          if (omask == 0) continue;
          const int node = __shfl_sync(0xffffffffu, en.x, 16 * q);
          const int first = __shfl_sync(0xffffffffu, v.t.x, 16 * q);
          const int nchild = __shfl_sync(0xffffffffu, v.t.y, 16 * q);
          if (first < 0) {
            if (lane == 0) W.leaf[nleaf] = make_int2(node, (int)omask);
            ++nleaf;
          } else {
            if (lane < nchild) W.st[sp + lane] = make_int2(first + lane, (int)omask);
            sp += nchild;
          }
        }
      }
      __syncwarp();
      for (int i = 0; i < nleaf; ++i) {
        // an opened leaf: x_a - x_b = r - (x_b - c), its particles in order
        const int2 en = W.leaf[i];
        const NodeF* f = nf + en.x;
        const float4 cm = __ldg(&f->cm);
        const int4 lt4 = __ldg(&f->t);
        const float r[3] = {(ph[0] - cm.x) + (pl[0] - __ldg(&f->q1.w)),
                            (ph[1] - cm.y) + (pl[1] - __ldg(&f->lo.w)),
                            (ph[2] - cm.z) + (pl[2] - __ldg(&f->hi.w))};
        const bool on = ((uint32_t)en.y >> tl) & 1u;
        const float4* pp = po + 2 * pair_base(lt4.z, en.x);
        const int npairs = (lt4.w + 1) >> 1;
        const int self = on && a32 >= lt4.z && a32 < lt4.z + lt4.w ? a32 - lt4.z : -1;
        const bool any_self = __any_sync(0xffffffffu, self >= 0);
        if (!on) continue;
        if (half == 0) npair += (uint32_t)lt4.w - (self >= 0 ? 1u : 0u);
        const float2 rx = f2(r[0]), ry = f2(r[1]), rz = f2(r[2]);
        for (int j = half; j < npairs; j += 2) {
          const float4 u = __ldg(pp + 2 * j), w = __ldg(pp + 2 * j + 1);
          const float2 dx = __fadd2_rn(rx, make_float2(-u.x, -u.y));
          const float2 dy = __fadd2_rn(ry, make_float2(-u.z, -u.w));
          const float2 dz = __fadd2_rn(rz, make_float2(-w.x, -w.y));
          float2 d2 = __ffma2_rn(dx, dx, f2(k32.eps2));
          d2 = __ffma2_rn(dy, dy, d2);
          d2 = __ffma2_rn(dz, dz, d2);
          float2 m = make_float2(w.z, w.w);
          if (any_self && self >= 0 && (self >> 1) == j) {  // the target itself: no force
            if (self & 1) {
              m.y = 0.f;
              d2.y = 1.f;
            } else {
              m.x = 0.f;
              d2.x = 1.f;
            }
          }
          const float2 inv = make_float2(rsqrt_ftz(d2.x), rsqrt_ftz(d2.y));
          const float2 fb = __fmul2_rn(m, __fmul2_rn(__fmul2_rn(inv, inv), inv));
          px = __ffma2_rn(fb, dx, px);
          py = __ffma2_rn(fb, dy, py);
          pz = __ffma2_rn(fb, dz, pz);
        }
      }
      __syncwarp();
    }
    if (sp > 0 && lane == 0) raise_flag(err, SPH_FLAG_CELL_OVERFLOW);
    nodes_used += used;
    pairs += npair;
    acc[0] -= px.x + px.y;
    acc[1] -= py.x + py.y;
    acc[2] -= pz.x + pz.y;
#pragma unroll
    for (int q = 0; q < 3; ++q) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], kTile32);
    if (valid && half == 0) {
      gx[a] = k32.Gs * acc[0];
      gy[a] = k32.Gs * acc[1];
      gz[a] = k32.Gs * acc[2];
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    nodes_used += __shfl_xor_sync(0xffffffffu, nodes_used, o);
    pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
  }
  if (lane == 0) {
    atomicAdd(stats, nodes_used);
    atomicAdd(stats + 1, pairs);
  }
}

inline int blocks_for(int64_t n, int sm, int threads) {
  int64_t b = (n + threads - 1) / threads;
  const int64_t cap = (int64_t)sm * 32;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

}  // namespace grav
}  // namespace sph

namespace {

int gfail(sph_ctx* ctx, cudaError_t e, const char* what) { return sph::cuda_fail(ctx, e, what); }

// Grow-only scratch of the gravity call.
int grav_scratch(sph_ctx* ctx, size_t bytes) {
  if (ctx->grav_bytes >= bytes) return SPH_OK;
  if (ctx->grav_buf) cudaFree(ctx->grav_buf);
  ctx->grav_buf = nullptr;
  ctx->grav_bytes = 0;
  cudaError_t e = cudaMalloc(&ctx->grav_buf, bytes);
  if (e != cudaSuccess) return gfail(ctx, e, "sph_gravity scratch");
  ctx->grav_bytes = bytes;
  return SPH_OK;
}

}  // namespace

extern "C" int sph_gravity(sph_ctx* ctx, sph_state* state, double G, double eps, double theta,
                           double* gx, double* gy, double* gz, int64_t* interactions,
                           sph_stream_t stream) {
  using sph::grav::Node;
  if (!ctx) return SPH_ERR_INVALID_ARG;
  if (!state) return sph::set_error(ctx, SPH_ERR_INVALID_ARG, "NULL state");
  const int64_t n = state->n;
  if (n < 0 || n > ctx->n_max)
    return sph::set_error(ctx, SPH_ERR_INVALID_ARG, "n = %lld outside [0, n_max]", (long long)n);
  if (!(theta >= 0.0) || !(eps >= 0.0) || !(G == G))
    return sph::set_error(ctx, SPH_ERR_INVALID_ARG, "theta and eps must be >= 0");
  for (int k = 0; k < 3; ++k)
    if (ctx->prm.periodic[k])
      return sph::set_error(ctx, SPH_ERR_INVALID_ARG,
                            "self-gravity needs open boundaries on every axis");
  if (n == 0) {  // nothing to read or write: the arrays may be NULL
    if (interactions) interactions[0] = interactions[1] = 0;
    return SPH_OK;
  }
  if (!gx || !gy || !gz) return sph::set_error(ctx, SPH_ERR_INVALID_ARG, "NULL output");
  const double* req[] = {state->x, state->y, state->z, state->vx, state->vy, state->vz,
                         state->vxh, state->vyh, state->vzh, state->h, state->m, state->u,
                         state->du_prev};
  for (const double* q : req)
    if (!q) return sph::set_error(ctx, SPH_ERR_INVALID_ARG, "a state array is NULL");
  if (!state->id) return sph::set_error(ctx, SPH_ERR_INVALID_ARG, "id is NULL");
  cudaStream_t st = (cudaStream_t)stream;
  sph::StateView in;
  in.x = state->x;
  in.y = state->y;
  in.z = state->z;
  in.vx = state->vx;
  in.vy = state->vy;
  in.vz = state->vz;
  in.vxh = state->vxh;
  in.vyh = state->vyh;
  in.vzh = state->vzh;
  in.h = state->h;
  in.m = state->m;
  in.u = state->u;
  in.du_prev = state->du_prev;
  in.id = state->id;
  // the library's grid and Morton sort (the state is reordered in place)
  sph::launch_grid(ctx, in, n, st);
  sph::launch_sort_gather(ctx, in, n, st);
  sph::launch_copy_state(in, ctx->s, n, st, ctx);
  ctx->have_lists = 0;
  ctx->have_density = ctx->have_iad = 0;
  sph::Grid g;
  cudaError_t e = cudaMemcpyAsync(&g, ctx->grid, sizeof(g), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return gfail(ctx, e, "sph_gravity grid");
  const int64_t n_occ = g.n_occ;
  const int bits = g.bits;
  // scratch: nodes (worst case n_occ per level), two code arrays, flags, scan
  const int64_t cap = n_occ * (bits + 1) + 1;
  const int64_t nparts = (n_occ + sph::scan::kScanItems - 1) / sph::scan::kScanItems + 1;
  const size_t off_code0 = sizeof(Node) * (size_t)cap;
  const size_t off_code1 = off_code0 + sizeof(uint32_t) * (size_t)n_occ;
  const size_t off_flag = off_code1 + sizeof(uint32_t) * (size_t)n_occ;
  const size_t off_idx = (off_flag + sizeof(int32_t) * (size_t)n_occ + 15) & ~(size_t)15;
  const size_t off_part = off_idx + sizeof(int64_t) * (size_t)(n_occ + 1);
  const size_t off_stats = off_part + sizeof(int64_t) * (size_t)nparts;
  const bool fp32 = ctx->prm.precision == SPH_FP32_MIXED;
  const size_t off_nf = (off_stats + 3 * sizeof(unsigned long long) + 127) & ~(size_t)127;
  const size_t off_po = off_nf + sizeof(sph::grav::NodeF) * (size_t)cap;
  const size_t bytes = off_po + (fp32 ? 2 * sizeof(float4) * (size_t)((n + n_occ) / 2 + 1) : 0);
  int rc = grav_scratch(ctx, bytes);
  if (rc != SPH_OK) return rc;
  char* base = (char*)ctx->grav_buf;
  Node* nodes = (Node*)base;
  uint32_t* code_a = (uint32_t*)(base + off_code0);
  uint32_t* code_b = (uint32_t*)(base + off_code1);
  int32_t* flag = (int32_t*)(base + off_flag);
  int64_t* idx = (int64_t*)(base + off_idx);
  int64_t* part = (int64_t*)(base + off_part);
  unsigned long long* stats = (unsigned long long*)(base + off_stats);
  int64_t* n_nodes = (int64_t*)(stats + 2);
  e = cudaMemsetAsync(stats, 0, 2 * sizeof(unsigned long long), st);
  if (e != cudaSuccess) return gfail(ctx, e, "sph_gravity");
  const int sm = ctx->sm_count;
  sph::grav::k_leaves<<<sph::grav::blocks_for(n_occ, sm, 128), 128, 0, st>>>(
      ctx->grid, ctx->occ, ctx->tbl_start, ctx->tbl_count, n_occ, code_a, nodes, in);
  ctx->launches += 1;
  int64_t coff = 0, m = n_occ, noff = n_occ;
  int l = bits - 1;
  for (; l >= 0 && m > sph::grav::kTopNodes; --l) {
    sph::grav::k_run_flags<<<sph::grav::blocks_for(m, sm, 256), 256, 0, st>>>(code_a, m, flag);
    sph::scan::exclusive_scan(flag, m, part, idx, st);
    int64_t npar = 0;
    e = cudaMemcpyAsync(&npar, idx + m, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return gfail(ctx, e, "sph_gravity tree level");
    sph::grav::k_parents<<<sph::grav::blocks_for(m, sm, 256), 256, 0, st>>>(
        code_a, flag, idx, m, coff, noff, code_b, nodes);
    sph::grav::k_parent_moments<<<sph::grav::blocks_for(npar, sm, 128), 128, 0, st>>>(
        ctx->grid, code_b, npar, m, coff, noff, l, nodes);
    ctx->launches += 6;
    uint32_t* t = code_a;
    code_a = code_b;
    code_b = t;
    coff = noff;
    noff += npar;
    m = npar;
  }
  sph::grav::k_top<<<1, sph::grav::kTopThreads, 0, st>>>(ctx->grid, code_a, code_b, m, coff, noff, l,
                                                         nodes, n_nodes);
  ctx->launches += 1;
  const int64_t tiles = (n + sph::grav::kTile32 - 1) / sph::grav::kTile32;
  int wb = (int)((tiles + sph::grav::kWalkWarps - 1) / sph::grav::kWalkWarps);
  if (wb > sm * 256) wb = sm * 256;
  sph::grav::NodeF* nf = (sph::grav::NodeF*)(base + off_nf);
  double L = 0.0;
  for (int ax = 0; ax < 3; ++ax) L = fmax(L, 1.001 * g.nc[ax] * g.cs[ax]);
  // states may lie anywhere in the double range: FP32 coordinates are scaled to
  // [0, 2) by a power of two (exact)
  sph::grav::Walk32Consts k32;
  k32.sc = !(L > 0.0) || !isfinite(L) ? 1.0 : ldexp(1.0, -ilogb(L));
  L *= k32.sc;
  k32.lx = g.lo[0];
  k32.ly = g.lo[1];
  k32.lz = g.lo[2];
  k32.theta = theta;
  k32.Gs = G * k32.sc * k32.sc;
  k32.eps2 = (float)((eps * k32.sc) * (eps * k32.sc));
  k32.th = (float)theta;
  k32.mb = (float)(4.0 * L * 5.9604644775390625e-8);  // 4 L 2^-24
  k32.aL = (float)(8.0 * L * 5.9604644775390625e-8);  // 8 L 2^-24
  sph::grav::k_nodes32<<<sph::grav::blocks_for(2 * n_occ, sm, 128), 128, 0, st>>>(
      nodes, n_nodes, g.lo[0], g.lo[1], g.lo[2], k32.sc, nf);
  if (fp32) {
    float4* po = (float4*)(base + off_po);
    sph::grav::k_leaf_pairs<<<sph::grav::blocks_for(16 * n_occ, sm, 128), 128, 0, st>>>(
        nodes, n_occ, in, k32.sc, po);
    sph::grav::k_walk32<<<wb, 32 * sph::grav::kWalkWarps, 0, st>>>(
        nodes, nf, po, n_nodes, in, n, k32, gx, gy, gz, stats, ctx->err);
    ctx->launches += 3;
  } else {
    const int64_t tiles64 = (n + sph::grav::kTile64 - 1) / sph::grav::kTile64;
    int wb64 = (int)((tiles64 + sph::grav::kWalkWarps - 1) / sph::grav::kWalkWarps);
    if (wb64 > sm * 256) wb64 = sm * 256;
    sph::grav::k_walk<<<wb64, 32 * sph::grav::kWalkWarps, 0, st>>>(
        nodes, nf, n_nodes, in, n, k32, G, eps * eps, gx, gy, gz, stats, ctx->err);
    ctx->launches += 2;
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return gfail(ctx, e, "sph_gravity launch");
  if (interactions) {
    unsigned long long h[2];
    e = cudaMemcpyAsync(h, stats, sizeof(h), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return gfail(ctx, e, "sph_gravity stats");
    interactions[0] = (int64_t)h[0];
    interactions[1] = (int64_t)h[1];
  }
  return SPH_OK;
}
