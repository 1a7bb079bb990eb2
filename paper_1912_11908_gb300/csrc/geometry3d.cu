// 3-D immersed-boundary pre-processing on the GPU (Sec. 3.2, Sec. 4.1-4.2;
// Appendix A's sphere in a cube): ray-casting classification of every node of
// a uniform lattice against a closed triangulated surface, IB / ghost tagging
// over the 6-neighbourhood, ordered node lists, and for every listed node the
// closest surface feature (face, edge or vertex) with its pseudo-normal.
//
// Compiled with -fmad=false: every decision and coordinate comes from IEEE
// basic operations and sqrt evaluated in a fixed order, so tags, lists and
// closest-feature records are reproducible bit for bit.  Face normals and
// the angle-weighted vertex pseudo-normals (Eq. 2, which needs acos) are
// formed once on the host when the body is created.
#include <cuda_runtime.h>

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <map>
#include <utility>
#include <vector>

#include "ibm.h"

extern "C" ibm_status ibm__noalloc_fail(ibm_status s, const char *msg);

namespace {

constexpr int B3 = 256;        // threads per block
constexpr uint8_t T_FLUID = IBM_TAG_FLUID, T_SOLID = IBM_TAG_SOLID, T_IB = IBM_TAG_IB, T_G1 = IBM_TAG_G1;

struct Lattice {
  int nx, ny, nz;
  double lo[3], d[3];
};

// exact per-face data of the closest-feature search: vertices, the entries of the barycentric normal equations and
// the squared edge lengths (the operations of evaluating them at every node, done once on the host)
struct FaceExact {
  double V[3][3];
  double a11, a12, a22, det;
  double ee[3];
};

constexpr int CL = 32;    // faces per cluster (Morton order of the centroids): one face per lane
constexpr int FPLANES = 6;

struct Mesh {
  int nv, ntri, ncl;
  const double *v;    // [nv][3]
  const int *tri;     // [ntri][3]
  const double *fn;   // [ntri][3] unit face normals
  const double *vn;   // [nv][3] unit angle-weighted vertex pseudo-normals
  const int *enb;     // [ntri][3] the face across edge k (vertices k, k+1), -1 if none
  const FaceExact *fx;// [ntri]
  const float4 *cl;   // [ncl][2] bounding box of a cluster's faces, widened by 1e-5 of the extent: lo, hi
  const float4 *fp;   // [FPLANES][ncl * CL] FP32 faces of the clusters: vertices, unit normal, the unit in-plane
                      // normals of the edges (inward), face index (bits; -1: padding), thickness and relative error
                      // of a thin face (0: not thin)
  float ext;          // largest coordinate magnitude of the mesh (at least 1e-12)
  double bb[6];       // axis-aligned bounding box: lo x, y, z, hi x, y, z
};

// node (i, j, k) of a node index (fewer than 2^31 nodes: 32-bit division)
__device__ __forceinline__ void node_ijk(const Lattice &L, int n, int ijk[3]) {
  const unsigned nxy = (unsigned)L.nx * (unsigned)L.ny, m = (unsigned)n;
  const unsigned k = m / nxy, r = m - k * nxy, j = r / (unsigned)L.nx;
  ijk[2] = (int)k;
  ijk[1] = (int)j;
  ijk[0] = (int)(r - j * (unsigned)L.nx);
}

__device__ __forceinline__ void node_xyz(const Lattice &L, int n, double P[3], int ijk[3]) {
  node_ijk(L, n, ijk);
  for (int a = 0; a < 3; a++) P[a] = L.lo[a] + ((double)ijk[a] + 0.5) * L.d[a];
}

// ---- classification (Sec. 3.2) over bit planes ------------------------------------------------------------------
// Rays along +x, +y and +z; a node is solid when at least two of its three crossing counts are odd and it lies in
// the surface's bounding box.  Whether the ray from a node crosses a face depends on the face's edge functions at
// the line's two transverse coordinates, the same for every node of the lattice line; only "ahead of the node", the
// sign of n.(a - P), depends on the node, and along a line that expression is monotone in the node's coordinate
// (each of its rounded operations is), so the nodes with the crossing ahead are the line's first t*, found by
// bisection with the node's own operations.  A crossing therefore toggles one bit -- the last node that has it ahead
// -- and a node's parity is the XOR of the bits at and beyond it.
//
// Layout: one bit per node, a word per 32 nodes along x (rows of pw words), one plane per ray axis; bit operations
// then vote and tag 32 nodes at a time.  The work per face is its projected area in lines instead of all lines times
// all faces: FP64, which bounds every exact geometric test on GB300 (2 lanes per SM and clock), is spent on the few
// lines in a face's own projected box.  Appendix A sphere, 1200 faces (ncu, cold caches): classification and lists
// 3.00 -> 0.16 ms at 256^3 nodes (k3_cross 0.11), 0.14 -> 0.055 ms at 40^3 (launches of 5-7 us each).
struct SubBox {
  int b0[3], n[3];  // nodes inside the bounding box along each axis: first index and count (n > 0)
};

// sign of the edge function e at P in the (u, v) projection, endpoints taken in increasing vertex index (the two
// faces sharing the edge see opposite values), a zero resolved by the symbolic shift of P by (eps, eps^2) in (u, v)
struct EdgeFn {
  double au, av, du, dv;
  int flip;
};
__device__ __forceinline__ EdgeFn edge_fn(const double *pa, int ia, const double *pb, int ib, int u, int v) {
  EdgeFn e;
  e.flip = 1;
  if (ib < ia) {
    const double *t = pa;
    pa = pb;
    pb = t;
    e.flip = -1;
  }
  e.au = pa[u];
  e.av = pa[v];
  e.du = pb[u] - pa[u];
  e.dv = pb[v] - pa[v];
  return e;
}
__device__ __forceinline__ int edge_sign(const EdgeFn &f, double Pu, double Pv) {
  const double e = f.du * (Pv - f.av) - f.dv * (Pu - f.au);
  int sg = e > 0.0 ? 1 : (e < 0.0 ? -1 : 0);
  if (sg == 0) sg = -f.dv > 0.0 ? 1 : (-f.dv < 0.0 ? -1 : 0);
  if (sg == 0) sg = f.du > 0.0 ? 1 : (f.du < 0.0 ? -1 : 0);
  return f.flip * sg;
}

// lattice index range of [lo, hi] along axis a, one node wider on each side, within the sub-box
__device__ __forceinline__ void index_range(const Lattice &L, const SubBox &B, int a, double lo, double hi, int &i0,
                                            int &i1) {
  const double first = (double)B.b0[a], last = (double)(B.b0[a] + B.n[a] - 1);
  const double x0 = floor((lo - L.lo[a]) / L.d[a] - 0.5) - 1.0, x1 = ceil((hi - L.lo[a]) / L.d[a] - 0.5) + 1.0;
  i0 = (int)fmin(fmax(x0, first), last + 1.0);
  i1 = (int)fmax(fmin(x1, last), first - 1.0);
}

// One (face, ray axis): its projected box in lattice lines and what the edge and plane tests need
struct CrossItem {
  EdgeFn e[3];
  double n[3], a[3];  // unnormalised normal and first vertex, in the order (u, v, axis)
  int u0, v0, nu, axis;
};

template <int axis>
__device__ __forceinline__ long long cross_item(const Lattice &L, const Mesh &m, const SubBox &B, int f, CrossItem &o) {
  constexpr int u = (axis + 1) % 3, v = (axis + 2) % 3;
  const int i0 = __ldg(m.tri + 3 * f), i1 = __ldg(m.tri + 3 * f + 1), i2 = __ldg(m.tri + 3 * f + 2);
  double a[3], b[3], c[3];
  for (int q = 0; q < 3; q++) {
    a[q] = __ldg(m.v + 3 * i0 + q);
    b[q] = __ldg(m.v + 3 * i1 + q);
    c[q] = __ldg(m.v + 3 * i2 + q);
  }
  int u0, u1, v0, v1;
  index_range(L, B, u, fmin(a[u], fmin(b[u], c[u])), fmax(a[u], fmax(b[u], c[u])), u0, u1);
  index_range(L, B, v, fmin(a[v], fmin(b[v], c[v])), fmax(a[v], fmax(b[v], c[v])), v0, v1);
  const double e1[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
  const double e2[3] = {c[0] - a[0], c[1] - a[1], c[2] - a[2]};
  const double nf[3] = {e1[1] * e2[2] - e1[2] * e2[1], e1[2] * e2[0] - e1[0] * e2[2], e1[0] * e2[1] - e1[1] * e2[0]};
  o.e[0] = edge_fn(a, i0, b, i1, u, v);
  o.e[1] = edge_fn(b, i1, c, i2, u, v);
  o.e[2] = edge_fn(c, i2, a, i0, u, v);
  o.n[0] = nf[u];
  o.n[1] = nf[v];
  o.n[2] = nf[axis];
  o.a[0] = a[u];
  o.a[1] = a[v];
  o.a[2] = a[axis];
  o.u0 = u0;
  o.v0 = v0;
  o.nu = u1 - u0 + 1;
  o.axis = axis;
  // a face parallel to the ray is not crossed
  return nf[axis] != 0.0 && o.nu > 0 && v1 >= v0 ? (long long)o.nu * (v1 - v0 + 1) : 0;
}

// Moller-Trumbore crossings: a block prepares 32 (face, axis) items, one per lane of its first warp, and its threads
// then take the items' lines one each (an FP64 warp instruction costs the same however few lanes are active, so both
// parts keep the lanes full; a warp per item spent 40 us on the items' set-up alone at 1200 faces).  gridDim.y blocks
// share the same items' lines.  A crossing toggles its bit in the axis' plane (XOR: independent of the order).
constexpr int XT = 128;
__global__ void __launch_bounds__(XT) k3_cross(Lattice L, Mesh m, SubBox B, int pw, unsigned *__restrict__ planes,
                                               long long plane_words) {
  __shared__ CrossItem item[32];
  __shared__ long long end[32];  // inclusive prefix sums of the items' lines
  if (threadIdx.x < 32) {
    const long long i = (long long)blockIdx.x * 32 + threadIdx.x;
    long long lines = 0;
    if (i < 3LL * m.ntri) {
      const int axis = (int)(i / m.ntri), f = (int)(i - (long long)axis * m.ntri);
      lines = axis == 0   ? cross_item<0>(L, m, B, f, item[threadIdx.x])
              : axis == 1 ? cross_item<1>(L, m, B, f, item[threadIdx.x])
                          : cross_item<2>(L, m, B, f, item[threadIdx.x]);
    }
    for (int o = 1; o < 32; o <<= 1) {
      const long long x = __shfl_up_sync(0xffffffffu, lines, o);
      if ((int)threadIdx.x >= o) lines += x;
    }
    end[threadIdx.x] = lines;
  }
  __syncthreads();
  const long long total = end[31];
  for (long long p = threadIdx.x + (long long)XT * blockIdx.y; p < total; p += (long long)XT * gridDim.y) {
    int it = 0;
    for (int s = 16; s > 0; s >>= 1)
      if (end[it + s - 1] <= p) it += s;  // the first item whose prefix sum exceeds p
    const CrossItem &c = item[it];
    const long long l = p - (it ? end[it - 1] : 0);
    const int dv = (int)(l / c.nu), iu = c.u0 + (int)(l - (long long)dv * c.nu), iv = c.v0 + dv, axis = c.axis;
    const int u = axis == 2 ? 0 : axis + 1, v = axis == 0 ? 2 : axis - 1;
    const double Pu = L.lo[u] + ((double)iu + 0.5) * L.d[u], Pv = L.lo[v] + ((double)iv + 0.5) * L.d[v];
    const int s0 = edge_sign(c.e[0], Pu, Pv);
    if (s0 == 0 || s0 != edge_sign(c.e[1], Pu, Pv) || s0 != edge_sign(c.e[2], Pu, Pv)) continue;
    // the line's first t* nodes have the crossing ahead: n.(a - P) of the sign of n_axis
    const double tu = c.n[0] * (c.a[0] - Pu), tv = c.n[1] * (c.a[1] - Pv), na = c.n[2], aa = c.a[2];
    const double La = L.lo[axis], Da = L.d[axis];
    const int first = B.b0[axis];
    auto ahead = [&](int t) {
      const double Q = La + ((double)(first + t) + 0.5) * Da;
      const double ta = na * (aa - Q);
      // the sum in coordinate order: x + y + z
      const double num = axis == 0 ? (ta + tu) + tv : axis == 1 ? (tv + ta) + tu : (tu + tv) + ta;
      return (num > 0.0 && na > 0.0) || (num < 0.0 && na < 0.0);
    };
    // bisection, begun around the crossing's position from one division
    int lo = 0, hi = B.n[axis];
    const double g = floor((aa + (tu + tv) / na - La) / Da - 0.5) - (double)first;
    const int gi = (int)fmin(fmax(g, 0.0), (double)hi);
    if (gi > 0 && gi - 1 < hi) {
      if (ahead(gi - 1)) lo = gi;
      else hi = gi - 1;
    }
    if (lo == gi && gi + 1 < hi && !ahead(gi + 1)) hi = gi + 1;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (ahead(mid)) lo = mid + 1;
      else hi = mid;
    }
    if (lo == 0) continue;
    const int at = first + lo - 1;
    const int x = axis == 0 ? at : axis == 1 ? iv : iu, y = axis == 0 ? iu : axis == 1 ? at : iv,
              z = axis == 0 ? iv : axis == 1 ? iu : at;
    atomicXor(planes + axis * plane_words + ((long long)z * L.ny + y) * pw + (x >> 5), 1u << (x & 31));
  }
}

// suffix XOR of n words w[0], w[stride], ...: SEG threads of a column (threadIdx.y) take a segment each, the segments
// behind a thread's own enter through shared memory; op(t, parity) receives every word's parity, from the last on
constexpr int SEG = 8;
template <class Op>
__device__ __forceinline__ void suffix_xor(const unsigned *w, long long stride, int n, bool live,
                                           unsigned (*part)[32], Op op) {
  const int per = (n + SEG - 1) / SEG, t0 = min(n, (int)threadIdx.y * per), t1 = min(n, t0 + per);
  unsigned x = 0;
  if (live) {
#pragma unroll 4
    for (int t = t0; t < t1; t++) x ^= w[t * stride];
  }
  part[threadIdx.y][threadIdx.x] = x;
  __syncthreads();
  if (!live) return;
  unsigned acc = 0;
  for (int s = threadIdx.y + 1; s < SEG; s++) acc ^= part[s][threadIdx.x];
#pragma unroll 4
  for (int t = t1 - 1; t >= t0; t--) {
    acc ^= w[t * stride];
    op(t, acc);
  }
}

// parities of the x and y rays in place: blocks [0, nyb) the y columns (a word column per threadIdx.x), the rest one
// thread per x row
__global__ void __launch_bounds__(32 * SEG) k3_parity_xy(Lattice L, SubBox B, int pw, unsigned *__restrict__ xb,
                                                         unsigned *__restrict__ yb, int nyb) {
  __shared__ unsigned part[SEG][32];
  const int w0 = B.b0[0] >> 5, nw = ((B.b0[0] + B.n[0] - 1) >> 5) - w0 + 1;
  if ((int)blockIdx.x < nyb) {
    const int col = blockIdx.x * 32 + threadIdx.x, k = col / nw;
    const bool live = k < B.n[2];
    unsigned *p = yb + ((long long)(B.b0[2] + (live ? k : 0)) * L.ny + B.b0[1]) * pw + w0 + (col - k * nw);
    suffix_xor(p, pw, B.n[1], live, part, [&](int t, unsigned par) { p[(long long)t * pw] = par; });
    return;
  }
  const unsigned r = (blockIdx.x - nyb) * (32u * SEG) + threadIdx.y * 32 + threadIdx.x, k = r / (unsigned)B.n[1];
  if (k >= (unsigned)B.n[2]) return;
  unsigned *p = xb + ((long long)(B.b0[2] + (int)k) * L.ny + B.b0[1] + (int)(r - k * (unsigned)B.n[1])) * pw + w0;
  unsigned carry = 0;
  for (int w = nw - 1; w >= 0; w--) {
    unsigned y = p[w];
    for (int s = 1; s < 32; s <<= 1) y ^= y >> s;  // bit i: XOR of the bits at and above i
    y ^= carry;
    p[w] = y;
    carry = y & 1u ? 0xffffffffu : 0u;
  }
}

// parity of the z rays and the vote: at least two of the three, inside the bounding box
__global__ void __launch_bounds__(32 * SEG) k3_vote(Lattice L, SubBox B, int pw, const unsigned *__restrict__ xb,
                                                    const unsigned *__restrict__ yb, const unsigned *__restrict__ zb,
                                                    unsigned *__restrict__ sb) {
  __shared__ unsigned part[SEG][32];
  const int w0 = B.b0[0] >> 5, x1 = B.b0[0] + B.n[0] - 1, nw = (x1 >> 5) - w0 + 1;
  const int col = blockIdx.x * 32 + threadIdx.x, j = col / nw, w = w0 + col - j * nw;
  const bool live = j < B.n[1];
  const unsigned lom = (w << 5) < B.b0[0] ? 0xffffffffu << (B.b0[0] & 31) : 0xffffffffu;
  const unsigned him = (w << 5) + 31 > x1 ? 0xffffffffu >> (31 - (x1 & 31)) : 0xffffffffu;
  const long long o = ((long long)B.b0[2] * L.ny + B.b0[1] + (live ? j : 0)) * pw + w, st = (long long)L.ny * pw;
  suffix_xor(zb + o, st, B.n[2], live, part, [&](int t, unsigned z) {
    const unsigned x = xb[o + t * st], y = yb[o + t * st];
    sb[o + t * st] = ((x & y) | (z & (x | y))) & lom & him;
  });
}

// Sec. 3.2 / Sec. 5 over the 6-neighbourhood, the 32 nodes of a word at a time: m[0] = IB (fluid node with a solid
// neighbour), m[1..3] = G1..G3 (solid node whose nearest non-solid node along a lattice line is 1..3 nodes away);
// returns the word's solid bits.  Nodes off the lattice are neither solid nor fluid.
__device__ __forceinline__ unsigned node_masks(const Lattice &L, int pw, const unsigned *__restrict__ sb,
                                               long long wi, unsigned m[4], int &w, int &row) {
  row = (int)(wi / pw);
  w = (int)(wi - (long long)row * pw);
  const int k = row / L.ny, j = row - k * L.ny;
  const unsigned tail = L.nx & 31 ? 0xffffffffu >> (32 - (L.nx & 31)) : 0xffffffffu;
  const unsigned vm = w == pw - 1 ? tail : 0xffffffffu;
  const unsigned S = sb[wi], F = ~S & vm;
  const unsigned Sl = w > 0 ? sb[wi - 1] : 0u, Sr = w < pw - 1 ? sb[wi + 1] : 0u;
  const unsigned Fl = w > 0 ? ~Sl : 0u, Fr = w < pw - 1 ? ~Sr & (w + 1 == pw - 1 ? tail : 0xffffffffu) : 0u;
  unsigned near_s = (S << 1 | Sl >> 31) | (S >> 1 | Sr << 31), near_f[3];
  for (int s = 1; s <= 3; s++) near_f[s - 1] = (F << s | Fl >> (32 - s)) | (F >> s | Fr << (32 - s));
  const long long py = pw, pz = (long long)L.ny * pw;
#pragma unroll
  for (int s = 1; s <= 3; s++) {
    const unsigned a = j >= s ? sb[wi - s * py] : vm, b = j + s < L.ny ? sb[wi + s * py] : vm;
    const unsigned c = k >= s ? sb[wi - s * pz] : vm, d = k + s < L.nz ? sb[wi + s * pz] : vm;
    near_f[s - 1] |= (~a | ~b | ~c | ~d) & vm;
    if (s == 1)
      near_s |= (j >= 1 ? a : 0u) | (j + 1 < L.ny ? b : 0u) | (k >= 1 ? c : 0u) | (k + 1 < L.nz ? d : 0u);
  }
  m[0] = F & near_s;
  m[1] = S & near_f[0];
  m[2] = S & near_f[1] & ~m[1];
  m[3] = S & near_f[2] & ~(m[1] | m[2]);
  return S;
}

// tags (zero = fluid on entry: only words with solid or IB nodes are written, a byte per lane) and per block the
// counts of IB, G1, G2, G3; one word per thread
__global__ void __launch_bounds__(B3) k3_tags(Lattice L, int pw, long long nwords, const unsigned *__restrict__ sb,
                                              uint8_t *__restrict__ tags, int *__restrict__ blockcounts) {
  __shared__ int wc[B3 / 32][4];
  const long long wi = (long long)blockIdx.x * B3 + threadIdx.x;
  const int lane = threadIdx.x & 31;
  unsigned m[4] = {0u, 0u, 0u, 0u}, S = 0u;
  int w = 0, row = 0;
  if (wi < nwords) S = node_masks(L, pw, sb, wi, m, w, row);
  for (unsigned todo = __ballot_sync(0xffffffffu, (S | m[0]) != 0u); todo; todo &= todo - 1) {
    const int src = __ffs(todo) - 1;
    const unsigned s = __shfl_sync(0xffffffffu, S, src);
    unsigned q[4];
    for (int t = 0; t < 4; t++) q[t] = __shfl_sync(0xffffffffu, m[t], src);
    const int x = (__shfl_sync(0xffffffffu, w, src) << 5) + lane, r = __shfl_sync(0xffffffffu, row, src);
    if (x < L.nx) {
      const unsigned b = 1u << lane;
      const uint8_t t = q[0] & b ? T_IB : q[1] & b ? T_G1 : q[2] & b ? T_G1 + 1 : q[3] & b ? T_G1 + 2
                        : s & b ? T_SOLID : T_FLUID;
      tags[(long long)r * L.nx + x] = t;
    }
  }
  for (int q = 0; q < 4; q++) {
    const int c = (int)__reduce_add_sync(0xffffffffu, (unsigned)__popc(m[q]));
    if (lane == 0) wc[threadIdx.x >> 5][q] = c;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    int s = 0;
    for (int t = 0; t < B3 / 32; t++) s += wc[t][threadIdx.x];
    blockcounts[4 * blockIdx.x + threadIdx.x] = s;
  }
}

// exclusive scan over the block's threads of one value per thread (sh: one int per warp); total receives the sum
__device__ __forceinline__ int block_scan(int x, int *sh, int &total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int inc = x;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) sh[warp] = inc;
  __syncthreads();
  int before = 0;
  total = 0;
  for (int t = 0; t < nw; t++) {
    if (t < warp) before += sh[t];
    total += sh[t];
  }
  __syncthreads();
  return before + inc - x;
}

// exclusive offsets of every block within each class's list, and the class totals (counts[0..3]); one block
__global__ void __launch_bounds__(1024) k3_scan(int nblk, int *__restrict__ blockcounts, int *__restrict__ counts) {
  __shared__ int sh[32];
  const int per = (nblk + 1023) / 1024, b0 = min(nblk, (int)threadIdx.x * per), b1 = min(nblk, b0 + per);
  for (int q = 0; q < 4; q++) {
    int s = 0, total;
    for (int b = b0; b < b1; b++) s += blockcounts[4 * b + q];
    int off = block_scan(s, sh, total);
    for (int b = b0; b < b1; b++) {
      const int x = blockcounts[4 * b + q];
      blockcounts[4 * b + q] = off;
      off += x;
    }
    if (threadIdx.x == 0) counts[q] = total;
  }
}

// listed nodes in row-major order, IB first, then G1, G2, G3; entries past cap are not written.  One word per
// thread, its masks formed again from the solid bits
__global__ void __launch_bounds__(B3) k3_scatter(Lattice L, int pw, long long nwords, const unsigned *__restrict__ sb,
                                                 const int *__restrict__ blockoff, const int *__restrict__ counts,
                                                 int *__restrict__ nodes, int cap) {
  __shared__ int sh[B3 / 32];
  const long long wi = (long long)blockIdx.x * B3 + threadIdx.x;
  unsigned m[4] = {0u, 0u, 0u, 0u};
  int w = 0, row = 0;
  if (wi < nwords) node_masks(L, pw, sb, wi, m, w, row);
  if (!__syncthreads_or((m[0] | m[1] | m[2] | m[3]) != 0u)) return;
  const int n0 = row * L.nx + (w << 5);
  int base = 0;
  for (int q = 0; q < 4; q++) {
    int total;
    int pos = base + blockoff[4 * blockIdx.x + q] + block_scan(__popc(m[q]), sh, total);
    for (unsigned b = m[q]; b; b &= b - 1, pos++)
      if (pos < cap) nodes[pos] = n0 + __ffs(b) - 1;
    base += counts[q];
  }
}

__device__ __forceinline__ double dot3(const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; }

// Sec. 4.1: closest point of face f to P -- the plane projection (barycentric normal equations) when it falls
// inside the face, else the nearest point of its three edges (an end vertex when the edge parameter clamps);
// fv receives the local vertex of a vertex feature
__device__ __forceinline__ double face_closest(const FaceExact &F, const double P[3], double q[3], int &fk, int &fe,
                                               int &fv) {
  double V[3][3];
  for (int k = 0; k < 3; k++)
    for (int d = 0; d < 3; d++) V[k][d] = F.V[k][d];
  const double *A = V[0];
  const double e1[3] = {V[1][0] - A[0], V[1][1] - A[1], V[1][2] - A[2]};
  const double e2[3] = {V[2][0] - A[0], V[2][1] - A[1], V[2][2] - A[2]};
  const double w[3] = {P[0] - A[0], P[1] - A[1], P[2] - A[2]};
  const double a11 = F.a11, a12 = F.a12, a22 = F.a22, det = F.det, b1 = dot3(w, e1), b2 = dot3(w, e2);
  const double s = (b1 * a22 - b2 * a12) / det, r = (a11 * b2 - a12 * b1) / det;
  fk = 0;
  fe = 0;
  fv = 0;
  if (s >= 0.0 && r >= 0.0 && s + r <= 1.0) {
    for (int d = 0; d < 3; d++) q[d] = A[d] + s * e1[d] + r * e2[d];
  } else {
    double dmin = INFINITY;
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const double *E0 = V[k], *E1 = V[(k + 1) % 3];
      const double ed[3] = {E1[0] - E0[0], E1[1] - E0[1], E1[2] - E0[2]};
      const double pw[3] = {P[0] - E0[0], P[1] - E0[1], P[2] - E0[2]};
      double u = dot3(pw, ed) / F.ee[k];
      int vert = -1;
      if (u <= 0.0) {
        u = 0.0;
        vert = k;
      } else if (u >= 1.0) {
        u = 1.0;
        vert = (k + 1) % 3;
      }
      const double x[3] = {E0[0] + u * ed[0], E0[1] + u * ed[1], E0[2] + u * ed[2]};
      const double dd[3] = {P[0] - x[0], P[1] - x[1], P[2] - x[2]};
      const double d2 = dot3(dd, dd);
      if (d2 < dmin) {
        dmin = d2;
        q[0] = x[0];
        q[1] = x[1];
        q[2] = x[2];
        fk = vert >= 0 ? IBM_FEATURE_VERTEX : IBM_FEATURE_EDGE;
        fe = k;
        fv = vert;
      }
    }
  }
  const double dq[3] = {P[0] - q[0], P[1] - q[1], P[2] - q[2]};
  return dot3(dq, dq);
}

// the closest so far of a lane's faces (f = 0x7fffffff: none)
struct Nearest {
  double d2, q[3];
  int f, fk, fe, fv;
};
// face f taken into account, the lowest index among equal distances (a call: inlined into the search of the survivors, its
// registers pushed the search's own into local memory)
__device__ __noinline__ void take_face(const FaceExact &F, int f, const double P[3], Nearest &b) {
  double q[3];
  int fk, fe, fv;
  const double d2 = face_closest(F, P, q, fk, fe, fv);
  if (d2 < b.d2 || (d2 == b.d2 && f < b.f)) {
    b.d2 = d2;
    for (int d = 0; d < 3; d++) b.q[d] = q[d];
    b.f = f;
    b.fk = fk;
    b.fe = fe;
    b.fv = fv;
  }
}

// the record of node n from the winning face's closest feature: its pseudo-normal (Sec. 4.2) is the face normal, the
// angle-weighted vertex normal (Eq. 2) or the normalised sum of the two faces' normals at an edge (Eq. 3)
__device__ __forceinline__ void write_record(const Mesh &m, int n, int f, int fk, int fe, int fv, const double q[3],
                                             ibm_closest3d *__restrict__ out) {
  double nn[3];
  if (fk == IBM_FEATURE_FACE) {
    for (int d = 0; d < 3; d++) nn[d] = m.fn[3 * f + d];
  } else if (fk == IBM_FEATURE_VERTEX) {
    const int v = m.tri[3 * f + fv];
    for (int d = 0; d < 3; d++) nn[d] = m.vn[3 * v + d];
  } else {
    const int g = m.enb[3 * f + fe];
    for (int d = 0; d < 3; d++) nn[d] = m.fn[3 * f + d] + (g >= 0 ? m.fn[3 * g + d] : 0.0);
    const double Ln = sqrt(dot3(nn, nn));
    if (Ln > 0.0)
      for (int d = 0; d < 3; d++) nn[d] = nn[d] / Ln;
  }
  ibm_closest3d o;
  o.node = n;
  o.tri = f;
  o.kind = fk;
  o.reserved = 0;
  for (int d = 0; d < 3; d++) {
    o.cp[d] = q[d];
    o.n[d] = nn[d];
  }
  *out = o;
}

// minimum over the warp (no NaN among the values: distances and infinities)
__device__ __forceinline__ float warp_min(float x) {
  for (int o = 16; o > 0; o >>= 1) x = fminf(x, __shfl_xor_sync(0xffffffffu, x, o));
  return x;
}

// FP32 bounds of the distance from P to the lane's face of cluster c: lb below and ub above the distance that the
// exact evaluation finds, by the margin mg (far above the FP32 rounding of coordinates and operations).  Every term
// is well conditioned whatever the face's shape: the distances to the three edge segments, the distance to the plane,
// and the signed in-plane distances to the edge lines, which say whether the projection falls inside, outside, or
// within the margin of an edge (then the plane's distance bounds from below only).
// A thin face's barycentric system is too flat for that to describe its FP64 solution, off by up to `error` times the
// farthest vertex' distance; but whatever the solution, the point it accepts lies in the face, whose points are within
// the face's thickness of its longest edge and no farther away than the farthest vertex.  (Never pruned and pruning
// nothing, the thin sides of a tube sent most nodes to the evaluation of all faces.)
__device__ __forceinline__ void face_bounds(const Mesh &m, int c, int lane, const float P[3], float mg, float &lb,
                                            float &ub, int &f) {
  const int i = c * CL + lane, n = m.ncl * CL;
  float r[4 * FPLANES];
#pragma unroll
  for (int p = 0; p < FPLANES; p++) {
    const float4 q = __ldg(m.fp + (size_t)p * n + i);
    r[4 * p] = q.x;
    r[4 * p + 1] = q.y;
    r[4 * p + 2] = q.z;
    r[4 * p + 3] = q.w;
  }
  f = __float_as_int(r[21]);
  float e2 = INFINITY, tin = INFINITY, w[3][3];
#pragma unroll
  for (int k = 0; k < 3; k++)
    for (int d = 0; d < 3; d++) w[k][d] = P[d] - r[3 * k + d];
#pragma unroll
  for (int k = 0; k < 3; k++) {
    const int k1 = (k + 1) % 3;
    const float ex = r[3 * k1] - r[3 * k], ey = r[3 * k1 + 1] - r[3 * k + 1], ez = r[3 * k1 + 2] - r[3 * k + 2];
    const float we = fmaf(w[k][0], ex, fmaf(w[k][1], ey, w[k][2] * ez)), ee = fmaf(ex, ex, fmaf(ey, ey, ez * ez));
    const float u = fminf(fmaxf(__fdividef(we, ee), 0.0f), 1.0f);  // (an edge of length 0: NaN -> 0)
    const float dx = fmaf(-u, ex, w[k][0]), dy = fmaf(-u, ey, w[k][1]), dz = fmaf(-u, ez, w[k][2]);
    e2 = fminf(e2, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
    tin = fminf(tin, fmaf(w[k][0], r[12 + 3 * k], fmaf(w[k][1], r[13 + 3 * k], w[k][2] * r[14 + 3 * k])));
  }
  const float de = sqrtf(e2), h = fabsf(fmaf(w[0][0], r[9], fmaf(w[0][1], r[10], w[0][2] * r[11])));
  const float dm = fminf(h, de);
  ub = (tin >= mg ? dm : de) + mg;
  lb = (tin >= -mg ? dm : de) - mg;
  if (r[22] != 0.0f) {
    float v2 = 0.0f;
#pragma unroll
    for (int k = 0; k < 3; k++) v2 = fmaxf(v2, fmaf(w[k][0], w[k][0], fmaf(w[k][1], w[k][1], w[k][2] * w[k][2])));
    const float W = sqrtf(v2);
    ub = fminf(W, fmaf(r[23], W, de)) + mg;
    lb = r[22] < INFINITY ? de - r[22] - mg : -INFINITY;
  }
  if (f < 0) lb = ub = INFINITY;
}

// Sec. 4.1-4.2: closest feature of every listed node.  The exact evaluation (FP64, IEEE operations in a fixed order,
// the lowest face index among equal distances) is needed only for the faces that FP32 bounds cannot exclude -- one to
// a few per node -- and an FP64 warp instruction costs the same however few lanes are active, so the two parts are
// split: (1) a warp per node finds the surviving faces by bounds, over clusters of 32 spatially sorted faces (one
// face per lane), nearest cluster first; (2) the block's (node, face) pairs are evaluated one per thread, all lanes
// busy, and each node's lexicographic (distance, face) minimum writes its record.  Sphere of 1200 faces, 256^3
// lattice: 9.54 -> 0.29 ms, 40^3 0.41 -> 0.024 ms (issue-bound: 30% FMA, 29% ALU, FP64 18% of the cycles); one warp
// per node evaluating every face within a bounding-sphere bound took its candidates through FP64 code in nearly empty
// warps.  Boxes of the clusters instead of spheres halved the clusters visited (0.58 -> 0.29 ms).
constexpr int PAIRS = B3, KEEP = 96, NODES = 12;  // pairs per batch, survivors per node, nodes per warp and batch

__global__ void __launch_bounds__(B3, 3) k3_closest(Lattice L, Mesh m, const int *__restrict__ nodes,
                                                 const int *__restrict__ counts, int cap, float mg,
                                                 ibm_closest3d *__restrict__ rec) {
  __shared__ int s_face[B3 / 32][KEEP];
  __shared__ float s_lb[B3 / 32][KEEP];
  __shared__ int p_entry[PAIRS], p_face[PAIRS], p_first[PAIRS], p_count[PAIRS];
  __shared__ double p_d2[PAIRS];
  __shared__ int npairs;
  const int total = min(cap, counts[0] + counts[1] + counts[2] + counts[3]);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // nodes per warp and batch: an even share of the blocks' rounds over the list
  const int warps = (int)gridDim.x * (B3 / 32), rounds = 1 + total / (warps * NODES);
  const int npw = 1 + total / (warps * rounds);
  const int batch = npw * (B3 / 32);
  const float lo[3] = {(float)L.lo[0], (float)L.lo[1], (float)L.lo[2]};
  const float dd[3] = {(float)L.d[0], (float)L.d[1], (float)L.d[2]};
  for (long long e0 = (long long)blockIdx.x * batch; e0 < total; e0 += (long long)gridDim.x * batch) {
    if (threadIdx.x == 0) npairs = 0;
    __syncthreads();
    for (int q = 0; q < npw; q++) {
      if (e0 + q * (B3 / 32) + warp >= total) break;
      const int e = (int)e0 + q * (B3 / 32) + warp;
      const int n = nodes[e];
      int ijk[3];
      node_ijk(L, n, ijk);
      float P[3];
      for (int a = 0; a < 3; a++) P[a] = fmaf((float)ijk[a] + 0.5f, dd[a], lo[a]);
      // distances to the clusters' boxes (the first 64 kept); the cluster of the nearest centre comes first: its
      // faces give the first upper bound
      auto box = [&](int c, float &centre) {
        const float4 l = __ldg(m.cl + 2 * c), h = __ldg(m.cl + 2 * c + 1);
        const float dx = fmaxf(fmaxf(l.x - P[0], P[0] - h.x), 0.0f), dy = fmaxf(fmaxf(l.y - P[1], P[1] - h.y), 0.0f),
                    dz = fmaxf(fmaxf(l.z - P[2], P[2] - h.z), 0.0f);
        const float cx = 0.5f * (l.x + h.x) - P[0], cy = 0.5f * (l.y + h.y) - P[1], cz = 0.5f * (l.z + h.z) - P[2];
        centre = fmaf(cx, cx, fmaf(cy, cy, cz * cz));
        return sqrtf(fmaf(dx, dx, fmaf(dy, dy, dz * dz))) - mg;
      };
      float near = INFINITY, kept0 = INFINITY, kept1 = INFINITY;
      int c0 = 0;
      for (int c = lane; c < m.ncl; c += 32) {
        float q;
        const float d = box(c, q);
        if (c < 32) kept0 = d;
        else if (c < 64) kept1 = d;
        if (q < near) {
          near = q;
          c0 = c;
        }
      }
      const float first_near = warp_min(near);
      c0 = __shfl_sync(0xffffffffu, c0, __ffs(__ballot_sync(0xffffffffu, near == first_near)) - 1);
      float ub = INFINITY;
      int cnt = 0;
      bool over = false;
      // keep the listed faces whose lower bound is within the current upper bound
      auto compact = [&]() {
        int kept = 0;
        for (int i0 = 0; i0 < cnt; i0 += 32) {
          const int i = i0 + lane;
          const bool ok = i < cnt && s_lb[warp][i] <= ub;
          const int face = ok ? s_face[warp][i] : 0;
          const float b = ok ? s_lb[warp][i] : 0.0f;
          __syncwarp();
          const unsigned bal = __ballot_sync(0xffffffffu, ok);
          if (ok) {
            const int at = kept + __popc(bal & ((1u << lane) - 1u));
            s_face[warp][at] = face;
            s_lb[warp][at] = b;
          }
          kept += __popc(bal);
          __syncwarp();
        }
        cnt = kept;
      };
      auto visit = [&](int c) {
        float lb, fu;
        int f;
        face_bounds(m, c, lane, P, mg, lb, fu, f);
        ub = fminf(ub, warp_min(fu));
        if (over) return;
        const bool ok = f >= 0 && lb <= ub;
        const unsigned bal = __ballot_sync(0xffffffffu, ok);
        const int more = __popc(bal);
        if (cnt + more > KEEP) compact();
        if (cnt + more > KEEP) {
          over = true;
          return;
        }
        if (ok) {
          const int at = cnt + __popc(bal & ((1u << lane) - 1u));
          s_face[warp][at] = f;
          s_lb[warp][at] = lb;
        }
        cnt += more;
        __syncwarp();
      };
      // every cluster but `but` whose box is within the current upper bound
      auto for_near = [&](int but, auto fn) {
        for (int b = 0; b < m.ncl; b += 32) {
          const int c = b + lane;
          float d = b == 0 ? kept0 : kept1, unused;
          if (b >= 64 && c < m.ncl) d = box(c, unused);
          for (unsigned todo = __ballot_sync(0xffffffffu, c < m.ncl && c != but && d <= ub); todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1;
            if (__shfl_sync(0xffffffffu, d, src) <= ub) fn(b + src);
          }
        }
      };
      visit(c0);
      for_near(c0, visit);
      int first = PAIRS;
      if (!over) {
        compact();
        if (lane == 0) first = atomicAdd(&npairs, cnt);
        first = __shfl_sync(0xffffffffu, first, 0);
      }
      if (!over && first + cnt <= PAIRS) {
        for (int i = lane; i < cnt; i += 32) {
          p_entry[first + i] = e;
          p_face[first + i] = s_face[warp][i];
          p_first[first + i] = first;
          p_count[first + i] = cnt;
        }
        __syncwarp();
        continue;
      }
      // more survivors than the batch has room for: the warp evaluates them itself (found once more by their bounds if
      // they were not kept -- all faces instead: 1.5 s for 64^3 nodes around 400,000 faces, most nodes having a hundred of
      // them as near as the bounds can tell)
      if (!over && lane == 0)
        for (int i = first; i < PAIRS; i++) p_entry[i] = -1;  // the part of the claim inside the list stays empty
      double X[3];
      node_xyz(L, n, X, ijk);
      Nearest near_face = {INFINITY, {0.0, 0.0, 0.0}, 0x7fffffff, 0, 0, 0};
      if (over) cnt = 0;
      auto evaluate_kept = [&]() {
        for (int i = lane; i < cnt; i += 32) {
          const int f = s_face[warp][i];
          take_face(m.fx[f], f, X, near_face);
        }
        cnt = 0;
        __syncwarp();
      };
      if (over) {
        for_near(-1, [&](int c) {
          float lb, fu;
          int f;
          face_bounds(m, c, lane, P, mg, lb, fu, f);
          const bool ok = f >= 0 && lb <= ub;
          const unsigned bal = __ballot_sync(0xffffffffu, ok);
          if (cnt + __popc(bal) > KEEP) evaluate_kept();
          if (ok) s_face[warp][cnt + __popc(bal & ((1u << lane) - 1u))] = f;
          cnt += __popc(bal);
          __syncwarp();
        });
      }
      evaluate_kept();
      double md = near_face.d2;
      int mf = near_face.f;
      for (int o = 16; o > 0; o >>= 1) {
        const double od = __shfl_xor_sync(0xffffffffu, md, o);
        const int of = __shfl_xor_sync(0xffffffffu, mf, o);
        if (od < md || (od == md && of < mf)) {
          md = od;
          mf = of;
        }
      }
      if (near_face.f == mf && mf != 0x7fffffff)
        write_record(m, n, mf, near_face.fk, near_face.fe, near_face.fv, near_face.q, rec + e);
      __syncwarp();
    }
    __syncthreads();
    const int t = threadIdx.x, np = min(npairs, PAIRS);
    const bool live = t < np && p_entry[t] >= 0;
    double y[3];
    int fk = 0, fe = 0, fv = 0, n = 0;
    if (live) {
      n = nodes[p_entry[t]];
      double X[3];
      int ijk[3];
      node_xyz(L, n, X, ijk);
      p_d2[t] = face_closest(m.fx[p_face[t]], X, y, fk, fe, fv);
    }
    __syncthreads();
    if (live) {
      const double d2 = p_d2[t];
      const int f = p_face[t];
      bool win = d2 < INFINITY;
      for (int i = p_first[t]; i < p_first[t] + p_count[t]; i++)
        if (p_d2[i] < d2 || (p_d2[i] == d2 && p_face[i] < f)) win = false;
      if (win) write_record(m, n, f, fk, fe, fv, y, rec + p_entry[t]);
    }
    __syncthreads();
  }
}

// host: unit face normals and angle-weighted vertex pseudo-normals (Eq. 2), in the order of the faces
void host_normals(int nv, const double *v, int ntri, const int *tri, std::vector<double> &fn, std::vector<double> &vn) {
  fn.assign((size_t)3 * ntri, 0.0);
  vn.assign((size_t)3 * nv, 0.0);
  auto dot = [](const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
  auto unit = [&](double *a) {
    const double Ln = std::sqrt(dot(a, a));
    if (Ln > 0.0) {
      a[0] = a[0] / Ln;
      a[1] = a[1] / Ln;
      a[2] = a[2] / Ln;
    }
  };
  for (int f = 0; f < ntri; f++) {
    const int *t = tri + 3 * f;
    const double *A = v + 3 * t[0], *B = v + 3 * t[1], *C = v + 3 * t[2];
    const double e1[3] = {B[0] - A[0], B[1] - A[1], B[2] - A[2]};
    const double e2[3] = {C[0] - A[0], C[1] - A[1], C[2] - A[2]};
    double *n = &fn[(size_t)3 * f];
    n[0] = e1[1] * e2[2] - e1[2] * e2[1];
    n[1] = e1[2] * e2[0] - e1[0] * e2[2];
    n[2] = e1[0] * e2[1] - e1[1] * e2[0];
    unit(n);
    for (int k = 0; k < 3; k++) {
      const double *O = v + 3 * t[k], *X = v + 3 * t[(k + 1) % 3], *Y = v + 3 * t[(k + 2) % 3];
      const double a[3] = {X[0] - O[0], X[1] - O[1], X[2] - O[2]};
      const double b[3] = {Y[0] - O[0], Y[1] - O[1], Y[2] - O[2]};
      const double cosv = dot(a, b) / std::sqrt(dot(a, a) * dot(b, b));
      const double ang = std::acos(std::fmax(-1.0, std::fmin(1.0, cosv)));  // interior angle at vertex t[k]
      for (int d = 0; d < 3; d++) vn[(size_t)3 * t[k] + d] += ang * n[d];
    }
  }
  for (int k = 0; k < nv; k++) unit(&vn[(size_t)3 * k]);
}

// Sec. 4.3-4.6 and Sec. 5 in 3-D: the interpolation cube around X over the cell centres and its weights --
// trilinear when all eight corners carry an allowed tag, otherwise 1 / r^2 over the allowed ones (a corner hit
// exactly takes all the weight); returns the corner mask
__device__ int cube_weights(const Lattice &L, const uint8_t *__restrict__ tags, const double X[3], unsigned allowed,
                            int o[3], double w[8]) {
  const int n[3] = {L.nx, L.ny, L.nz};
  for (int a = 0; a < 3; a++) o[a] = (int)floor((X[a] - L.lo[a]) / L.d[a] - 0.5);
  int mask = 0;
  for (int b = 0; b < 8; b++) {
    const int ci = o[0] + (b & 1), cj = o[1] + (b >> 1 & 1), ck = o[2] + (b >> 2);
    w[b] = 0.0;
    if (ci < 0 || ci >= n[0] || cj < 0 || cj >= n[1] || ck < 0 || ck >= n[2]) continue;
    if (allowed & (1u << tags[((long long)ck * n[1] + cj) * n[0] + ci])) mask |= 1 << b;
  }
  if (mask == 255) {
    double f[3];
    for (int a = 0; a < 3; a++) {
      const double c0 = L.lo[a] + ((double)o[a] + 0.5) * L.d[a];
      f[a] = (X[a] - c0) / L.d[a];
    }
    for (int b = 0; b < 8; b++) {
      const double wx = (b & 1) ? f[0] : 1.0 - f[0];
      const double wy = (b >> 1 & 1) ? f[1] : 1.0 - f[1];
      const double wz = (b >> 2) ? f[2] : 1.0 - f[2];
      w[b] = wx * wy * wz;
    }
  } else if (mask != 0) {
    double inv[8];
    int hit = -1;
    for (int b = 0; b < 8; b++) inv[b] = 0.0;
    for (int b = 0; b < 8 && hit < 0; b++) {
      if (!(mask >> b & 1)) continue;
      const int idx[3] = {o[0] + (b & 1), o[1] + (b >> 1 & 1), o[2] + (b >> 2)};
      double r2 = 0.0;
      for (int a = 0; a < 3; a++) {
        const double r = X[a] - (L.lo[a] + ((double)idx[a] + 0.5) * L.d[a]);
        r2 = r2 + r * r;
      }
      if (r2 == 0.0) hit = b;
      else inv[b] = 1.0 / r2;
    }
    if (hit >= 0) {
      w[hit] = 1.0;
    } else {
      double sum = 0.0;
      for (int b = 0; b < 8; b++)
        if (mask >> b & 1) sum += inv[b];
      for (int b = 0; b < 8; b++)
        if (mask >> b & 1) w[b] = inv[b] / sum;
    }
  }
  return mask;
}

// one stencil per listed node (IB first, then G1..G3, as listed): boundary point P' = X - xi_node n on the
// tangent plane through the closest point, probe one cell diagonal h beyond an IB node, mirror image point of a
// ghost node (at least dmin / 2 from P'), pushed out by dmin up to three times while the cube has no valid
// corner; a node left without one counts in *nerr
__global__ void __launch_bounds__(B3) k3_stencils(Lattice L, const uint8_t *__restrict__ tags,
                                                  const int *__restrict__ nodes, const int *__restrict__ counts,
                                                  int cap, const ibm_closest3d *__restrict__ rec, double h,
                                                  double dmin, ibm_stencil3d *__restrict__ out,
                                                  int *__restrict__ nerr) {
  const int c0 = counts[0], c1 = counts[1], c2 = counts[2];
  const int total = min(cap, c0 + c1 + c2 + counts[3]);
  const int e = blockIdx.x * B3 + threadIdx.x;
  if (e >= total) return;
  const int kind = e < c0 ? 0 : e < c0 + c1 ? 1 : e < c0 + c1 + c2 ? 2 : 3;
  const ibm_closest3d r = rec[e];
  double X[3];
  int ijk[3];
  node_xyz(L, nodes[e], X, ijk);
  const double xi_node = (X[0] - r.cp[0]) * r.n[0] + (X[1] - r.cp[1]) * r.n[1] + (X[2] - r.cp[2]) * r.n[2];
  double b[3];
  for (int a = 0; a < 3; a++) b[a] = X[a] - xi_node * r.n[a];
  double xi_probe;
  if (kind == 0) {
    xi_probe = xi_node + h;
  } else {
    xi_probe = -xi_node;
    if (xi_probe < 0.5 * dmin) xi_probe = 0.5 * dmin;
  }
  const unsigned allowed = kind == 0 ? (1u << T_FLUID) : ((1u << T_FLUID) | (1u << T_IB));
  ibm_stencil3d s;
  int o[3] = {0, 0, 0}, mask = 0, nstep = 0;
  for (;;) {
    double P[3];
    for (int a = 0; a < 3; a++) P[a] = b[a] + xi_probe * r.n[a];
    mask = cube_weights(L, tags, P, allowed, o, s.w);
    if (mask != 0 || nstep == 3) break;
    xi_probe = xi_probe + dmin;
    nstep++;
  }
  if (mask == 0) atomicAdd(nerr, 1);
  s.node = nodes[e];
  s.kind = kind;
  s.region = r.kind;
  s.nstep = nstep;
  s.i0 = o[0];
  s.j0 = o[1];
  s.k0 = o[2];
  s.mask = mask;
  for (int a = 0; a < 3; a++) {
    s.n[a] = r.n[a];
    s.b[a] = b[a];
  }
  s.xi_node = xi_node;
  s.xi_probe = xi_probe;
  out[e] = s;
}

// Sec. 6 (Eq. 9) in 3-D: the probe of each triangle one cell diagonal out along its normal from its centroid
// (mn: per triangle the centroid and the unit normal, 6 doubles), pushed out by dmin up to three times while its
// cube has no fluid corner; the record's b is the centroid, xi_probe the probe distance, node the triangle
__global__ void __launch_bounds__(B3) k3_surface_stencils(Lattice L, const uint8_t *__restrict__ tags,
                                                          const double *__restrict__ mn, int ntri, double h,
                                                          double dmin, ibm_stencil3d *__restrict__ out) {
  const int f = blockIdx.x * B3 + threadIdx.x;
  if (f >= ntri) return;
  const double m[3] = {mn[6 * f], mn[6 * f + 1], mn[6 * f + 2]}, n[3] = {mn[6 * f + 3], mn[6 * f + 4], mn[6 * f + 5]};
  ibm_stencil3d s;
  double xi = h;
  int o[3] = {0, 0, 0}, mask = 0, nstep = 0;
  for (int st = 0; st <= 3; st++) {
    const double P[3] = {m[0] + xi * n[0], m[1] + xi * n[1], m[2] + xi * n[2]};
    mask = cube_weights(L, tags, P, 1u << T_FLUID, o, s.w);
    if (mask) break;
    if (st < 3) {
      xi = xi + dmin;
      nstep++;
    }
  }
  s.node = f;
  s.kind = 0;
  s.region = IBM_FEATURE_FACE;
  s.nstep = nstep;
  s.i0 = o[0];
  s.j0 = o[1];
  s.k0 = o[2];
  s.mask = mask;
  for (int a = 0; a < 3; a++) {
    s.n[a] = n[a];
    s.b[a] = m[a];
  }
  s.xi_node = 0.0;
  s.xi_probe = xi;
  out[f] = s;
}

}  // namespace

struct ibm_body3d {
  Mesh m{};
  char *mem = nullptr;       // mesh data on the device
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  Lattice L{};
  long long nn = 0;          // lattice nodes of the last classification
  int pw = 0;                // words per lattice row of the bit planes
  long long nwords = 0;      // words per bit plane
  int nblk = 0, cap = 0;
  unsigned *bits = nullptr;  // four bit planes: crossings (then parities) of the x, y and z rays, solid nodes
  uint8_t *tags = nullptr;
  int *blockcounts = nullptr, *counts = nullptr, *nodes = nullptr;
  ibm_closest3d *rec = nullptr;
  bool classified = false;
};

static ibm_status cuda_fail(cudaError_t e) { return ibm__noalloc_fail(IBM_ECUDA, cudaGetErrorString(e)); }

static void free_lattice(ibm_body3d *b) {
  cudaFree(b->bits);
  cudaFree(b->tags);
  cudaFree(b->blockcounts);
  cudaFree(b->counts);
  cudaFree(b->nodes);
  cudaFree(b->rec);
  b->bits = nullptr;
  b->tags = nullptr;
  b->blockcounts = b->counts = b->nodes = nullptr;
  b->rec = nullptr;
  b->nn = 0;
}

extern "C" ibm_status ibm_body3d_create(const double *verts, int nverts, const int32_t *tris, int ntris,
                                        void *cuda_stream, ibm_body3d **out) {
  if (!out || !verts || !tris || nverts < 4 || ntris < 4) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_create: bad mesh");
  *out = nullptr;
  for (int k = 0; k < 3 * ntris; k++)
    if (tris[k] < 0 || tris[k] >= nverts) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_create: vertex index out of range");
  std::vector<double> fn, vn;
  host_normals(nverts, verts, ntris, tris, fn, vn);
  // the face across each edge: the first face (in index order) holding the reversed directed edge
  std::map<std::pair<int, int>, int> first;
  for (int f = 0; f < ntris; f++)
    for (int k = 0; k < 3; k++) first.emplace(std::make_pair(tris[3 * f + k], tris[3 * f + (k + 1) % 3]), f);
  std::vector<int> enb((size_t)3 * ntris, -1);
  for (int f = 0; f < ntris; f++)
    for (int k = 0; k < 3; k++) {
      auto it = first.find(std::make_pair(tris[3 * f + (k + 1) % 3], tris[3 * f + k]));
      if (it != first.end()) enb[(size_t)3 * f + k] = it->second;
    }
  // closest-feature search: exact per-face data, and FP32 faces in clusters of 32 along a Morton curve through the
  // centroids, so that a cluster is compact; bounding boxes widened by 1e-5 of the mesh's extent
  double ext = 0.0, blo[3] = {INFINITY, INFINITY, INFINITY}, bhi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (int k = 0; k < nverts; k++)
    for (int a = 0; a < 3; a++) {
      blo[a] = std::min(blo[a], verts[3 * k + a]);
      bhi[a] = std::max(bhi[a], verts[3 * k + a]);
    }
  for (int a = 0; a < 3; a++) ext = std::max(ext, std::max(std::fabs(blo[a]), std::fabs(bhi[a])));
  ext = std::max(ext, 1e-12);  // (FP32 squares of smaller distances would underflow)
  const double margin = 1e-5 * ext;
  std::vector<FaceExact> fx((size_t)ntris);
  std::vector<std::pair<uint32_t, int>> order((size_t)ntris);
  for (int f = 0; f < ntris; f++) {
    const double *V[3] = {verts + 3 * tris[3 * f], verts + 3 * tris[3 * f + 1], verts + 3 * tris[3 * f + 2]};
    FaceExact &x = fx[f];
    auto dot = [](const double *a, const double *b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
    double ed[3][3], e2[3];
    for (int k = 0; k < 3; k++)
      for (int d = 0; d < 3; d++) {
        x.V[k][d] = V[k][d];
        ed[k][d] = V[(k + 1) % 3][d] - V[k][d];
      }
    for (int d = 0; d < 3; d++) e2[d] = V[2][d] - V[0][d];
    x.a11 = dot(ed[0], ed[0]);
    x.a12 = dot(ed[0], e2);
    x.a22 = dot(e2, e2);
    x.det = x.a11 * x.a22 - x.a12 * x.a12;
    for (int k = 0; k < 3; k++) x.ee[k] = dot(ed[k], ed[k]);
    uint32_t key = 0;
    for (int a = 0; a < 3; a++) {
      const double c = (V[0][a] + V[1][a] + V[2][a]) / 3.0, w = bhi[a] - blo[a];
      const double t = w > 0.0 ? (c - blo[a]) / w : 0.0;
      const uint32_t g = t > 0.0 ? (uint32_t)std::min(1023.0, t * 1024.0) : 0u;
      for (int bit = 0; bit < 10; bit++) key |= (g >> bit & 1u) << (3 * bit + a);
    }
    order[f] = std::make_pair(key, f);
  }
  std::sort(order.begin(), order.end());
  const int ncl = (ntris + CL - 1) / CL;
  std::vector<float4> cl((size_t)2 * ncl), fp((size_t)FPLANES * ncl * CL);
  for (int c = 0; c < ncl; c++) {
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    const int i0 = c * CL, i1 = std::min(ntris, i0 + CL);
    for (int i = i0; i < i1; i++)
      for (int k = 0; k < 3; k++)
        for (int a = 0; a < 3; a++) {
          lo[a] = std::min(lo[a], fx[order[i].second].V[k][a]);
          hi[a] = std::max(hi[a], fx[order[i].second].V[k][a]);
        }
    for (int i = i0; i < i0 + CL; i++) {
      float r[4 * FPLANES] = {};
      int f = -1;
      if (i < i1) {
        f = order[i].second;
        const FaceExact &x = fx[f];
        const double *n = &fn[(size_t)3 * f];
        for (int k = 0; k < 3; k++) {
          const int k1 = (k + 1) % 3;
          const double e[3] = {x.V[k1][0] - x.V[k][0], x.V[k1][1] - x.V[k][1], x.V[k1][2] - x.V[k][2]};
          const double len = std::sqrt(x.ee[k]), il = len > 0.0 ? 1.0 / len : 0.0;
          const double in[3] = {n[1] * e[2] - n[2] * e[1], n[2] * e[0] - n[0] * e[2], n[0] * e[1] - n[1] * e[0]};
          for (int a = 0; a < 3; a++) {
            r[3 * k + a] = (float)x.V[k][a];
            r[12 + 3 * k + a] = (float)(in[a] * il);
          }
        }
        for (int a = 0; a < 3; a++) r[9 + a] = (float)n[a];
        // sin^2 of the angle at the first vertex below 1e-8 (thin): the FP64 barycentric solution may be off by more
        // than the margin.  With u = 2^-53, w the vertices' distances and the solution's s, t in [0, 1], each of its
        // products carries at most 13 u |w| |e|^3 and det 24 u |e|^4: the point is off by less than 150 u max|w| / sin^2.
        // Thickness: the height over the longest edge, |e1| |e2| sin / longest, rounding of det included; no bound
        // (infinity) where that is not a number
        const double aa = x.a11 * x.a22;
        if (!(x.det >= 1e-8 * aa)) {
          const double longest = std::max(x.ee[0], std::max(x.ee[1], x.ee[2]));
          const double h = 1.01 * std::sqrt((std::max(x.det, 0.0) + 1e-14 * aa) / longest);
          const double sin2 = x.det / aa - 1e-14;
          r[22] = h > 0.0 ? std::max((float)h, FLT_MIN) : x.a11 == 0.0 || x.a22 == 0.0 ? FLT_MIN : INFINITY;
          r[23] = sin2 > 0.0 ? (float)std::min(2e-14 / sin2, 1.0) : 1.0f;
        }
      }
      std::memcpy(&r[21], &f, sizeof f);
      for (int p = 0; p < FPLANES; p++)
        fp[(size_t)p * ncl * CL + i] = make_float4(r[4 * p], r[4 * p + 1], r[4 * p + 2], r[4 * p + 3]);
    }
    cl[2 * c] = make_float4((float)(lo[0] - margin), (float)(lo[1] - margin), (float)(lo[2] - margin), 0.f);
    cl[2 * c + 1] = make_float4((float)(hi[0] + margin), (float)(hi[1] + margin), (float)(hi[2] + margin), 0.f);
  }
  ibm_body3d *b = new ibm_body3d();
  b->m.nv = nverts;
  b->m.ntri = ntris;
  b->m.ncl = ncl;
  b->m.ext = (float)ext;
  for (int a = 0; a < 3; a++) {
    b->m.bb[a] = blo[a];
    b->m.bb[3 + a] = bhi[a];
  }
  const size_t sv = (size_t)3 * nverts * sizeof(double), st = (size_t)3 * ntris * sizeof(int),
               sf = (size_t)3 * ntris * sizeof(double);
  auto up = [](size_t x) { return (x + 255) & ~(size_t)255; };
  const size_t sfx = fx.size() * sizeof(FaceExact), scl = cl.size() * sizeof(float4), sfp = fp.size() * sizeof(float4);
  const size_t total = up(sv) * 2 + up(st) * 2 + up(sf) + up(sfx) + up(scl) + up(sfp);
  cudaError_t e = cudaMalloc(&b->mem, total);
  if (e != cudaSuccess) {
    delete b;
    return ibm__noalloc_fail(IBM_ENOMEM, "ibm_body3d_create: device allocation failed");
  }
  char *p = b->mem;
  double *dv = (double *)p;
  p += up(sv);
  double *dvn = (double *)p;
  p += up(sv);
  int *dt = (int *)p;
  p += up(st);
  int *den = (int *)p;
  p += up(st);
  double *dfn = (double *)p;
  p += up(sf);
  FaceExact *dfx = (FaceExact *)p;
  p += up(sfx);
  float4 *dcl = (float4 *)p;
  p += up(scl);
  float4 *dfp = (float4 *)p;
  if (cuda_stream) {
    b->stream = (cudaStream_t)cuda_stream;
  } else {
    e = cudaStreamCreate(&b->stream);
    b->own_stream = e == cudaSuccess;
  }
  if (e == cudaSuccess) e = cudaMemcpy(dv, verts, sv, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dvn, vn.data(), sv, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dt, tris, st, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(den, enb.data(), st, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dfn, fn.data(), sf, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dfx, fx.data(), sfx, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dcl, cl.data(), scl, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dfp, fp.data(), sfp, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    ibm_body3d_destroy(b);
    return cuda_fail(e);
  }
  b->m.v = dv;
  b->m.vn = dvn;
  b->m.tri = dt;
  b->m.enb = den;
  b->m.fn = dfn;
  b->m.fx = dfx;
  b->m.cl = dcl;
  b->m.fp = dfp;
  *out = b;
  return IBM_OK;
}

extern "C" ibm_status ibm_body3d_classify(ibm_body3d *b, const ibm_grid3d *g) {
  if (!b || !g || g->nx < 1 || g->ny < 1 || g->nz < 1) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_classify: bad grid");
  const long long nn = (long long)g->nx * g->ny * g->nz;
  if (nn > (1LL << 31) - 1) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_classify: more than 2^31 - 1 nodes");
  for (int a = 0; a < 3; a++)
    if (!(g->hi[a] > g->lo[a])) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_classify: empty domain");
  Lattice L;
  L.nx = g->nx;
  L.ny = g->ny;
  L.nz = g->nz;
  const int nd[3] = {g->nx, g->ny, g->nz};
  for (int a = 0; a < 3; a++) {
    L.lo[a] = g->lo[a];
    L.d[a] = (g->hi[a] - g->lo[a]) / (double)nd[a];
  }
  // listed nodes lie within three nodes of the bounding box
  long long cap = 1;
  for (int a = 0; a < 3; a++) {
    long long i0 = (long long)std::floor((b->m.bb[a] - L.lo[a]) / L.d[a] - 0.5) - 4;
    long long i1 = (long long)std::ceil((b->m.bb[3 + a] - L.lo[a]) / L.d[a] - 0.5) + 4;
    i0 = std::max(0LL, i0);
    i1 = std::min((long long)nd[a] - 1, i1);
    cap *= std::max(0LL, i1 - i0 + 1);
  }
  cap = std::max(1LL, std::min(cap, nn));
  cudaError_t e = cudaSuccess;
  const bool same = nn == b->nn && (int)cap == b->cap && g->nx == b->L.nx && g->ny == b->L.ny && g->nz == b->L.nz;
  if (!same) {
    e = cudaStreamSynchronize(b->stream);
    if (e != cudaSuccess) return cuda_fail(e);
    free_lattice(b);
    b->pw = (g->nx + 31) / 32;
    b->nwords = (long long)b->pw * g->ny * g->nz;
    b->nblk = (int)((b->nwords + B3 - 1) / B3);
    if (e == cudaSuccess) e = cudaMalloc(&b->bits, (size_t)4 * b->nwords * sizeof(unsigned));
    if (e == cudaSuccess) e = cudaMalloc(&b->tags, (size_t)nn);
    if (e == cudaSuccess) e = cudaMalloc(&b->blockcounts, (size_t)4 * b->nblk * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->counts, 4 * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->nodes, (size_t)cap * sizeof(int));
    if (e == cudaSuccess) e = cudaMalloc(&b->rec, (size_t)cap * sizeof(ibm_closest3d));
    if (e != cudaSuccess) {
      free_lattice(b);
      return ibm__noalloc_fail(IBM_ENOMEM, "ibm_body3d_classify: device allocation failed");
    }
    b->nn = nn;
    b->cap = (int)cap;
  }
  b->L = L;
  int dev = 0, nsm = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  // nodes inside the bounding box along each axis, by the nodes' own coordinates (non-decreasing in the index)
  SubBox B;
  bool any = true;
  for (int a = 0; a < 3; a++) {
    auto first = [&](auto outside) {  // first index that is not outside (n if none)
      int lo = 0, hi = nd[a];
      while (lo < hi) {
        const int mid = lo + (hi - lo) / 2;
        if (outside(L.lo[a] + ((double)mid + 0.5) * L.d[a])) lo = mid + 1;
        else hi = mid;
      }
      return lo;
    };
    B.b0[a] = first([&](double x) { return x < b->m.bb[a]; });
    B.n[a] = first([&](double x) { return !(x > b->m.bb[3 + a]); }) - B.b0[a];
    any = any && B.n[a] > 0;
  }
  unsigned *xb = b->bits, *yb = xb + b->nwords, *zb = yb + b->nwords, *sb = zb + b->nwords;
  cudaMemsetAsync(b->bits, 0, (size_t)4 * b->nwords * sizeof(unsigned), b->stream);
  cudaMemsetAsync(b->tags, T_FLUID, (size_t)nn, b->stream);
  if (any) {
    // 32 (face, axis) items per block; few faces have many lines each, shared by several blocks
    const int items = (int)((3LL * b->m.ntri + 31) / 32);
    k3_cross<<<dim3(items, std::max(1, std::min(1024, 4 * nsm / items))), XT, 0, b->stream>>>(L, b->m, B, b->pw, b->bits,
                                                                                             b->nwords);
    const int nw = ((B.b0[0] + B.n[0] - 1) >> 5) - (B.b0[0] >> 5) + 1;
    const int nyb = (int)(((long long)nw * B.n[2] + 31) / 32);
    const int nxb = (int)(((long long)B.n[1] * B.n[2] + 32 * SEG - 1) / (32 * SEG));
    k3_parity_xy<<<nyb + nxb, dim3(32, SEG), 0, b->stream>>>(L, B, b->pw, xb, yb, nyb);
    k3_vote<<<(int)(((long long)nw * B.n[1] + 31) / 32), dim3(32, SEG), 0, b->stream>>>(L, B, b->pw, xb, yb, zb, sb);
  }
  k3_tags<<<b->nblk, B3, 0, b->stream>>>(L, b->pw, b->nwords, sb, b->tags, b->blockcounts);
  k3_scan<<<1, 1024, 0, b->stream>>>(b->nblk, b->blockcounts, b->counts);
  k3_scatter<<<b->nblk, B3, 0, b->stream>>>(L, b->pw, b->nwords, sb, b->blockcounts, b->counts, b->nodes, b->cap);
  float mg = 0.0f;
  for (int a = 0; a < 3; a++) mg = std::max(mg, (float)std::max(std::fabs(g->lo[a]), std::fabs(g->hi[a])));
  mg = 1e-5f * b->m.ext + 2e-6f * mg;
  k3_closest<<<nsm * 3, B3, 0, b->stream>>>(L, b->m, b->nodes, b->counts, b->cap, mg, b->rec);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e);
  b->classified = true;
  return IBM_OK;
}

extern "C" ibm_status ibm_body3d_get(ibm_body3d *b, int what, void *dst, size_t bytes) {
  if (!b || !dst) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_get: NULL argument");
  if (!b->classified) return ibm__noalloc_fail(IBM_ESTATE, "ibm_body3d_get: not classified");
  cudaError_t e = cudaStreamSynchronize(b->stream);
  if (e != cudaSuccess) return cuda_fail(e);
  int cnt[4];
  e = cudaMemcpy(cnt, b->counts, sizeof(cnt), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e);
  const long long total = (long long)cnt[0] + cnt[1] + cnt[2] + cnt[3];
  const int n = (int)std::min<long long>(total, b->cap);
  switch (what) {
    case IBM_3D_TAGS:
      if (bytes < (size_t)b->nn) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_get: dst too small");
      e = cudaMemcpy(dst, b->tags, (size_t)b->nn, cudaMemcpyDeviceToHost);
      break;
    case IBM_3D_COUNTS:
      if (bytes < sizeof(cnt)) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_get: dst too small");
      std::memcpy(dst, cnt, sizeof(cnt));
      break;
    case IBM_3D_NODES:
      if (bytes < (size_t)n * sizeof(int32_t)) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_get: dst too small");
      if (n) e = cudaMemcpy(dst, b->nodes, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost);
      break;
    case IBM_3D_CLOSEST:
      if (bytes < (size_t)n * sizeof(ibm_closest3d)) return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_get: dst too small");
      if (n) e = cudaMemcpy(dst, b->rec, (size_t)n * sizeof(ibm_closest3d), cudaMemcpyDeviceToHost);
      break;
    default:
      return ibm__noalloc_fail(IBM_EINVAL, "ibm_body3d_get: unknown quantity");
  }
  if (e != cudaSuccess) return cuda_fail(e);
  if (total > b->cap) return ibm__noalloc_fail(IBM_ECAPACITY, "ibm_body3d_get: more listed nodes than the capacity");
  return IBM_OK;
}

extern "C" ibm_status ibm_body3d_destroy(ibm_body3d *b) {
  if (!b) return IBM_OK;
  if (b->stream) cudaStreamSynchronize(b->stream);
  free_lattice(b);
  cudaFree(b->mem);
  if (b->own_stream) cudaStreamDestroy(b->stream);
  delete b;
  return IBM_OK;
}

// The 3-D flow solver's view of a classification: enqueue the stencils of the listed nodes (k3_stencils) on the
// body's stream, with h the probe distance and dmin the push-out step, into out (capacity b->cap entries);
// *nerr (device) receives the number of nodes without a valid corner.  Returns the device tags and per-class
// counts and the list capacity.
ibm_status ibm__body3d_stencils(ibm_body3d *b, double h, double dmin, ibm_stencil3d *out, int *nerr,
                                const uint8_t **tags, const int **counts, int *cap) {
  if (!b || !b->classified) return ibm__noalloc_fail(IBM_ESTATE, "3-D stencils: body not classified");
  k3_stencils<<<(b->cap + B3 - 1) / B3, B3, 0, b->stream>>>(b->L, b->tags, b->nodes, b->counts, b->cap, b->rec, h,
                                                           dmin, out, nerr);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e);
  *tags = b->tags;
  *counts = b->counts;
  *cap = b->cap;
  return IBM_OK;
}

int ibm__body3d_capacity(const ibm_body3d *b) { return b ? b->cap : 0; }

// The force probes of the 3-D flow solver (k3_surface_stencils) on the body's stream.
ibm_status ibm__surface3d_stencils(ibm_body3d *b, const double *mn, int ntri, double h, double dmin,
                                   ibm_stencil3d *out) {
  if (!b || !b->classified) return ibm__noalloc_fail(IBM_ESTATE, "3-D surface probes: body not classified");
  if (ntri > 0)
    k3_surface_stencils<<<(ntri + B3 - 1) / B3, B3, 0, b->stream>>>(b->L, b->tags, mn, ntri, h, dmin, out);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? IBM_OK : cuda_fail(e);
}
