// abp_big.cu -- the phased form of the force call, for walkers that share a
// grid (multiple-walker runs) or that are too large for one shared-memory
// walker group. One MD step is three launches over all such walkers, six on a
// step that deposits:
//
//   k_big_cn       a1, coordination numbers: the A x B pair sum split over
//                  CTAs by chunks of B (kBigChunk entries); each CTA writes
//                  dCN/dx of its B entries, its partial CN and A gradients,
//                  and whether its share of the walker's atoms is finite
//   k_big_cvs      a1 (other CVs, partial sums combined in chunk order) and
//                  a2: every walker's hill height from the grid as it was
//                  before any deposit of the step (Jacobi order); on a step
//                  without deposits a4 as well
//   k_big_deposit  a3: the hills; shared grids add them to the FP64 shadow
//                  with atomics (order-independent up to FP64 rounding), own
//                  grids with the two-sum update of the fused form
//   k_big_refresh  shared grids: FP32 fields = FP64 shadow split into
//                  value + compensation (about 48 bits kept)
//   k_big_lookup   a4 after all deposits
//   k_big_force    a5, and in a closed loop the move of the atoms
//
// Each may start while the one before it ends (launch_chained). 32 walkers on a
// shared 256^3 grid, 200 x 10,000 pairs each, 10 closed-loop steps: 1739 us
// with a CTA per 1024 B entries (2.1 an SM), six launches a step and a look-up
// per 256 atoms; 1121 us now, 91 us of a step's 112 in the pair kernel.
//
// FP32_COMP grids only. The paper's bias routine is the serial counterpart
// (one CPU rank), SI "Minimization of Interprocess Communications".
#include <cuda_runtime.h>

#include <vector>

#include "abp_device.cuh"
#include "abp_launch.h"
#include "abp_md.cuh"

namespace abp {

namespace {

constexpr int kBigThreads = 256;
constexpr int kBigCnThreads = 64;  // k_big_cn: small CTAs, so that the last SM's share is small too
constexpr int kBigJB = 6;  // B entries a thread (pair kernel, 32 x 200 x 10,000 pairs: 96.5 us with 4, 91 with 6)
constexpr int kBigChunk = kBigCnThreads * kBigJB;
constexpr int kBigForceThreads = 128;
constexpr int kStencilPerBlock = 2048;

__host__ __device__ constexpr int fixed_bytes_f() { return (int)((sizeof(GroupFixed<float>) + 31) & ~(size_t)31); }

__host__ __device__ inline size_t up256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

// Per-walker scratch of the phased form (in the walker's jscratch):
//   BigHead | jA[na] | jB[nb] | a5 term tables
// for the walker's (single) COORD CV; jA/jB hold dCN/dx per list entry. Its
// CTAs' partial sums (in bpart): s[nchunk][2] | bad[nchunk] | g[nchunk][na][3].
struct BigHead {
  float sh[kMaxCv], sl[kMaxCv];
  float com_u[kMaxCv][3];
  float dih_g[kMaxCv][4][3];
  int da[kMaxCv], dc[kMaxCv], ic_log[kMaxCv];
  float df[kMaxCv];
  float hf;
  int dep, bad, flags;
  float dv[kMaxCv];  // dV_b/ds after the step's deposits
  double h;
};

__host__ __device__ inline int big_cn_index(const WalkerDev &wd) {
  for (int k = 0; k < wd.g.d; ++k)
    if (wd.cv[k].type == ABP_CV_COORD) return k;
  return -1;
}

__host__ __device__ inline int big_nchunks(const WalkerDev &wd) {
  int k = big_cn_index(wd);
  return k < 0 ? 0 : (wd.cv[k].nb + kBigChunk - 1) / kBigChunk;
}

struct BigLayout {
  size_t head, jA, jB, terms, nterm, total;
};

struct BigParts {
  float *s;   // [nchunk][2]
  int *bad;   // [nchunk]
  float *g;   // [nchunk][na][3]
};
__host__ __device__ inline BigParts big_parts(void *p, int nc) {
  BigParts P;
  P.s = static_cast<float *>(p);
  P.bad = reinterpret_cast<int *>(P.s + 2 * nc);
  P.g = reinterpret_cast<float *>(P.bad + nc);
  return P;
}

__host__ __device__ inline BigLayout big_layout(const WalkerDev &wd) {
  BigLayout L;
  int k = big_cn_index(wd);
  int na = k < 0 ? 0 : wd.cv[k].na, nb = k < 0 ? 0 : wd.cv[k].nb;
  L.head = 0;
  L.jA = up256(sizeof(BigHead));
  L.jB = L.jA + (size_t)na * 16;
  // per atom, its a5 terms (big_atom_terms) and their count
  L.terms = up256(L.jB + (size_t)nb * 16);
  L.nterm = up256(L.terms + (size_t)wd.natoms * kAtomTerms * 4);
  L.total = up256(L.nterm + (size_t)wd.natoms);
  return L;
}

// Term codes of the force phase: kind | k << 3 | list position << 5.
enum { kTermComA = 0, kTermComB = 1, kTermDih = 2, kTermCnA = 3, kTermCnB = 4 };

int big_atom_terms(const WalkerDev &hd, const abp_walker_desc *d, std::vector<int32_t> &terms,
                   std::vector<uint8_t> &cnt) {
  const int n = hd.natoms;
  terms.assign((size_t)n * kAtomTerms, 0);
  cnt.assign((size_t)n, 0);
  auto add = [&](int atom, int kind, int k, int pos) -> int {
    if (atom < 0 || atom >= n || cnt[atom] >= kAtomTerms || pos >= (1 << 26)) return -1;
    terms[(size_t)atom * kAtomTerms + cnt[atom]] = kind | (k << 3) | (pos << 5);
    cnt[atom] += 1;
    return 0;
  };
  // CV by CV, list A before list B: the order in which a5 adds them
  for (int k = 0; k < hd.g.d; ++k) {
    const abp_cv_desc &c = d->cv[k];
    const bool com = c.type == ABP_CV_COM_DIST, cn = c.type == ABP_CV_COORD;
    if (!com && !cn && c.type != ABP_CV_DIHEDRAL) return -1;
    const int na = c.type == ABP_CV_DIHEDRAL ? 4 : c.n_a;
    for (int i = 0; i < na; ++i)
      if (add(c.idx_a[i], com ? kTermComA : cn ? kTermCnA : kTermDih, k, i)) return -1;
    if (com || cn)
      for (int i = 0; i < c.n_b; ++i)
        if (add(c.idx_b[i], com ? kTermComB : kTermCnB, k, i)) return -1;
  }
  return 0;
}

size_t big_scratch_bytes(const WalkerDev &hd) { return big_layout(hd).total; }
size_t big_part_bytes(const WalkerDev &hd) {
  const int k = big_cn_index(hd), nc = big_nchunks(hd);
  return k < 0 ? 0 : (size_t)nc * (12 + (size_t)hd.cv[k].na * 12);
}
size_t big_terms_offset(const WalkerDev &hd) { return big_layout(hd).terms; }
size_t big_nterm_offset(const WalkerDev &hd) { return big_layout(hd).nterm; }
int big_cn_count(const WalkerDev &hd) {
  int n = 0;
  for (int k = 0; k < hd.g.d; ++k) n += hd.cv[k].type == ABP_CV_COORD;
  return n;
}
int big_chunks(const WalkerDev &hd) { return big_nchunks(hd); }

// ---------------------------------------------------------------- k_big_cn

// Minimum image d - L rint(d / L) with rint formed on the FMA pipe: adding
// and subtracting 1.5 2^23 rounds d / L to the nearest integer exactly for
// |d / L| < 2^22 (ties go to even, where either image has the same length).
__device__ __forceinline__ float min_image_rn(float d, float L, float invL) {
  const float M = 12582912.0f;
  const float t = __fsub_rn(__fmaf_rn(d, invL, M), M);
  return __fmaf_rn(-L, t, d);
}

// 1 / x for x >= 1 (infinity gives 0): one MUFU instruction.
__device__ __forceinline__ float rcp_ge1(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The A gradients of a block of 8 A atoms (x 3 components, this lane's part)
// summed over the warp by a reduce-scatter: three exchange levels halve the
// atoms a lane keeps (8, 4, 2, 1), two more add the rest; lane 4 q holds atom
// q's sums, which it stores.
__device__ __forceinline__ void reduce_block_grads(float (&v)[24], int lane, int n, float *out) {
#pragma unroll
  for (int o = 16, m = 12; o >= 4; o >>= 1, m >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < 12; ++i)
      if (i < m) {
        const float keep = up ? v[m + i] : v[i], send = up ? v[i] : v[m + i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
  }
#pragma unroll
  for (int o = 2; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 3; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
  const int q = lane >> 2;
  if ((lane & 3) == 0 && q < n)
#pragma unroll
    for (int i = 0; i < 3; ++i) out[3 * q + i] = v[i];
}

// A block of 8 A atoms (n of them valid) against the thread's kBigJB B
// entries. MASK: pairs with an A or B atom past the end count nothing. The
// switch values of an A atom, of at most kBigJB together, are added to a
// compensated sum that starts at kBigJB (three additions give the exact error).
template <bool PBC, bool MASK>
__device__ __forceinline__ void big_block(const float4 *As, int n, const float (&xj)[kBigJB], const float (&yj)[kBigJB],
                                          const float (&zj)[kBigJB], const float (&mj)[kBigJB], float (&gxj)[kBigJB],
                                          float (&gyj)[kBigJB], float (&gzj)[kBigJB], float k2, const float *box,
                                          const float *ibox, float &sacc, float &scomp, float (&gi)[24]) {
#pragma unroll
  for (int ii = 0; ii < 8; ++ii) {
    const float4 a = As[MASK && ii >= n ? 0 : ii];
    float g0 = 0.f, g1 = 0.f, g2 = 0.f, part = 0.f;
#pragma unroll
    for (int jj = 0; jj < kBigJB; ++jj) {
      float dx = a.x - xj[jj], dy = a.y - yj[jj], dz = a.z - zj[jj];
      if (PBC) {
        dx = min_image_rn(dx, box[0], ibox[0]);
        dy = min_image_rn(dy, box[1], ibox[1]);
        dz = min_image_rn(dz, box[2], ibox[2]);
      }
      const float q = (dx * dx + dy * dy + dz * dz) * k2;
      const float q2 = q * q;
      float sw = rcp_ge1(__fmaf_rn(q2, q, 1.f));
      if (MASK) sw *= ii < n ? mj[jj] : 0.f;
      part += sw;
      const float gf = q2 * (sw * sw);
      g0 += gf * dx;
      g1 += gf * dy;
      g2 += gf * dz;
      gxj[jj] += gf * dx;
      gyj[jj] += gf * dy;
      gzj[jj] += gf * dz;
    }
    const float t = __fadd_rn(sacc, part), z = __fsub_rn(t, sacc);
    scomp = __fadd_rn(scomp, __fsub_rn(part, z));
    sacc = t;
    gi[3 * ii] = g0;
    gi[3 * ii + 1] = g1;
    gi[3 * ii + 2] = g2;
  }
}

// One CTA: the A x (one chunk of B) pairs of one walker's CN. The A atoms are
// read from shared memory, each thread holds kBigJB B entries and their
// gradients. Bound by the FP32 issue: 18 operations a pair, 9 for a minimum
// image, ~6 for the sums and exchanges.
template <bool PBC>
__device__ __forceinline__ void big_cn_body(const BigItem &it, const CvDev &c, const float4 *x, float4 *As, float *lig) {
  const WalkerDev *wd = it.wd;
  const int na = c.na, nb = c.nb;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5, nwarps = kBigCnThreads / 32;
  const float k2 = (float)c.inv_r0sq, c6 = -6.f * k2;
  const float box[3] = {(float)c.box[0], (float)c.box[1], (float)c.box[2]};
  const float ibox[3] = {(float)c.inv_box[0], (float)c.inv_box[1], (float)c.inv_box[2]};
  const int j0 = it.chunk * kBigChunk;
  float xj[kBigJB], yj[kBigJB], zj[kBigJB], gxj[kBigJB], gyj[kBigJB], gzj[kBigJB], mj[kBigJB];
#pragma unroll
  for (int jj = 0; jj < kBigJB; ++jj) {
    const int j = j0 + jj * kBigCnThreads + t;
    const bool ok = j < nb;
    const float4 p = x[c.ib[ok ? j : 0]];
    xj[jj] = p.x;
    yj[jj] = p.y;
    zj[jj] = p.z;
    mj[jj] = ok ? 1.f : 0.f;
    gxj[jj] = gyj[jj] = gzj[jj] = 0.f;
  }
  float sacc = (float)kBigJB, scomp = 0.f;
  float *mylig = lig + warp * na * 3;
  const bool fullj = j0 + kBigChunk <= nb;
  for (int i0 = 0; i0 < na; i0 += 8) {
    const int n = min(8, na - i0);
    float gi[24];
    if (fullj && n == 8)
      big_block<PBC, false>(As + i0, n, xj, yj, zj, mj, gxj, gyj, gzj, k2, box, ibox, sacc, scomp, gi);
    else
      big_block<PBC, true>(As + i0, n, xj, yj, zj, mj, gxj, gyj, gzj, k2, box, ibox, sacc, scomp, gi);
    reduce_block_grads(gi, lane, n, mylig + 3 * i0);
  }
  const BigLayout L = big_layout(*wd);
  const BigParts P = big_parts(wd->bpart, big_nchunks(*wd));
  float4 *jB = reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(wd->jscratch) + L.jB);
#pragma unroll
  for (int jj = 0; jj < kBigJB; ++jj) {
    const int j = j0 + jj * kBigCnThreads + t;
    if (j < nb) jB[j] = make_float4(-c6 * gxj[jj], -c6 * gyj[jj], -c6 * gzj[jj], 0.f);
  }
  // this chunk's CN as hi + lo: lanes by butterfly, warps in order
  float h[1], l[1];
  two_sum<float>(__fsub_rn(sacc, (float)kBigJB), scomp, h[0], l[0]);
  warp_sum_ff<1>(h, l);
  __shared__ float wsum[kBigCnThreads / 32][2];
  if (lane == 0) {
    wsum[warp][0] = h[0];
    wsum[warp][1] = l[0];
  }
  __syncthreads();
  if (t == 0) {
    float sh = wsum[0][0], sl = wsum[0][1];
    for (int w = 1; w < nwarps; ++w) ff_add<float>(sh, sl, wsum[w][0], wsum[w][1]);
    P.s[2 * it.chunk] = sh;
    P.s[2 * it.chunk + 1] = sl;
  }
  float *part_g = P.g + (size_t)it.chunk * na * 3;
  for (int q = t; q < na * 3; q += kBigCnThreads) {
    float acc = lig[q];
    for (int w = 1; w < nwarps; ++w) acc += lig[w * na * 3 + q];
    part_g[q] = c6 * acc;
  }
}

__global__ void __launch_bounds__(kBigCnThreads, 6) k_big_cn(const BigItem *items, const void *coords,
                                                          const long long *coff, long long step_off) {
  extern __shared__ __align__(32) unsigned char smem[];
  const BigItem it = items[blockIdx.x];
  const WalkerDev *wd = it.wd;
  const CvDev &c = wd->cv[big_cn_index(*wd)];
  chain_wait();
  const float4 *x = reinterpret_cast<const float4 *>(coords) + coff[it.widx] + step_off;
  float4 *As = reinterpret_cast<float4 *>(smem);
  float *lig = reinterpret_cast<float *>(As + c.na);  // [warps][na][3]
  for (int i = threadIdx.x; i < c.na; i += kBigCnThreads) As[i] = x[c.ia[i]];
  // this CTA's share of the walker's atoms: all finite?
  const int nc = big_nchunks(*wd);
  const int lo = (int)((long long)wd->natoms * it.chunk / nc), hi = (int)((long long)wd->natoms * (it.chunk + 1) / nc);
  int bad = 0;
  for (int i = lo + (int)threadIdx.x; i < hi; i += kBigCnThreads) {
    const float4 p = x[i];
    bad |= (isfinite(p.x) && isfinite(p.y) && isfinite(p.z)) ? 0 : 1;
  }
  bad = __syncthreads_or(bad);  // (and the A atoms are in place)
  if (threadIdx.x == 0) big_parts(wd->bpart, nc).bad[it.chunk] = bad;
  if (c.pbc)
    big_cn_body<true>(it, c, x, As, lig);
  else
    big_cn_body<false>(it, c, x, As, lig);
}

// ---------------------------------------------------------------- k_big_cvs

__device__ __forceinline__ Grp big_group() {
  Grp g;
  g.G = blockDim.x;
  g.gid = 0;
  g.t = threadIdx.x;
  g.lane = threadIdx.x & 31;
  g.warp = threadIdx.x >> 5;
  g.nwarps = blockDim.x >> 5;
  return g;
}

__device__ void big_load_desc(const Grp &g, GroupFixed<float> *fx, const WalkerDev *wdp) {
  const int *s = reinterpret_cast<const int *>(wdp);
  int *d = reinterpret_cast<int *>(&fx->wd);
  for (int i = g.t; i < (int)(sizeof(WalkerDev) / 4); i += g.G) d[i] = s[i];
  g.sync();
  if (g.t < kMaxCv) {
    const CvDev &c = fx->wd.cv[g.t];
    fx->ia[g.t] = c.ia;
    fx->ib[g.t] = c.ib;
    fx->wa[g.t] = c.wa;
    fx->wb[g.t] = c.wb;
  }
  if (g.t == 0) {
    fx->flags = 0;
    fx->clamped = 0;
  }
  g.sync();
}

// Centre-of-mass distance with compensated arithmetic, by the whole CTA: each
// weighted offset w (x - r_G) is split exactly into hi + lo (the difference by
// two_sum, the product's error by fma; w times the difference's low part,
// tiny, rounded once), summed as hi + lo pairs, and |d| is taken in hi + lo
// (com_finish_ff). Groups spread over a large box (as a group of environment
// atoms is) otherwise lose the ~1e-8 relative accuracy a hill a few grid
// spacings wide needs. Part 1: every warp's sums to part[warp][6][2].
__device__ __forceinline__ void big_com_part(const Grp &g, const CvDev &c, const float4 *xs, float (*part)[6][2]) {
  const float4 ra = xs[c.ia[0]], rb = xs[c.ib[0]];
  float h[6] = {0, 0, 0, 0, 0, 0}, l[6] = {0, 0, 0, 0, 0, 0};
  auto acc = [&](int q, float w, float x, float r) {
    float dh, dl;
    two_sum<float>(x, -r, dh, dl);  // x - r exactly
    float p = __fmul_rn(w, dh);
    float e = __fmaf_rn(w, dl, __fmaf_rn(w, dh, -p));
    ff_add<float>(h[q], l[q], p, e);
  };
  for (int i = g.t; i < c.na; i += g.G) {
    float w = c.wa[i];
    float4 p = xs[c.ia[i]];
    acc(0, w, p.x, ra.x);
    acc(1, w, p.y, ra.y);
    acc(2, w, p.z, ra.z);
  }
  for (int i = g.t; i < c.nb; i += g.G) {
    float w = c.wb[i];
    float4 p = xs[c.ib[i]];
    acc(3, w, p.x, rb.x);
    acc(4, w, p.y, rb.y);
    acc(5, w, p.z, rb.z);
  }
  warp_sum_ff<6>(h, l);
  if (g.lane == 0)
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      part[g.warp][q][0] = h[q];
      part[g.warp][q][1] = l[q];
    }
}
// Part 2, by one warp: lane q < 6 adds the warps' sums of component q in warp
// order, lane 0 finishes.
__device__ __forceinline__ void big_com_end(const Grp &g, GroupFixed<float> *fx, int k, const float4 *xs,
                                            const float (*part)[6][2]) {
  const CvDev &c = fx->wd.cv[k];
  float h = 0.f, l = 0.f;
  if (g.lane < 6)
    for (int w = 0; w < g.nwarps; ++w) ff_add<float>(h, l, part[w][g.lane][0], part[w][g.lane][1]);
  float hh[6], ll[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    hh[q] = __shfl_sync(0xffffffffu, h, q);
    ll[q] = __shfl_sync(0xffffffffu, l, q);
  }
  if (g.lane != 0) return;
  const float4 ra = xs[c.ia[0]], rb = xs[c.ib[0]];
  const float a0[3] = {ra.x, ra.y, ra.z}, b0[3] = {rb.x, rb.y, rb.z};
  float s, sl;
  const int fl = com_finish_ff(c, a0, hh, ll, b0, hh + 3, ll + 3, s, sl, fx->com_u[k]);
  fx->sh[k] = s;
  fx->sl[k] = sl;
  if (fl) atomicOr(&fx->flags, fl);
}

// a4 of a walker whose CVs are in fx: V and dV/ds to its head and state.
__device__ __forceinline__ void big_lookup(const Grp &g, GroupFixed<float> *fx, BigHead *head, long long step) {
  const GroupLayout none{};
  interp_step<float, false>(g, fx, none, nullptr);
  const WalkerDev &wd = fx->wd;
  if (g.t == 0) {
    for (int k = 0; k < kMaxCv; ++k) head->dv[k] = k < wd.g.d ? fx->dvds[k] : 0.f;
    WalkerState st;
    for (int k = 0; k < 3; ++k) {
      st.s[k] = k < wd.g.d ? (double)fx->sh[k] + (double)fx->sl[k] : 0.0;
      st.dV[k] = k < wd.g.d ? (double)fx->dV[k] : 0.0;
    }
    st.V = (double)fx->V;
    st.flags = fx->flags;
    st.pad = 0;
    st.step = step;
    *wd.state = st;
  }
}

// One CTA per walker: CVs, axis state, height; hill record to the head; with
// `look` (no walker deposits this step) the look-up too.
__global__ void __launch_bounds__(kBigThreads) k_big_cvs(const BigItem *walkers, const void *coords,
                                                         const long long *coff, long long step_off, long long step,
                                                         DepositLog log, DevCounters *ctr, int look) {
  extern __shared__ __align__(32) unsigned char smem[];
  Grp g = big_group();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  const BigItem it = walkers[blockIdx.x];
  big_load_desc(g, fx, it.wd);
  chain_wait();
  const WalkerDev &wd = fx->wd;
  const float4 *x = reinterpret_cast<const float4 *>(coords) + coff[it.widx] + step_off;
  unsigned char *js = reinterpret_cast<unsigned char *>(wd.jscratch);
  BigHead *head = reinterpret_cast<BigHead *>(js);
  const int kc = big_cn_index(wd), nc = big_nchunks(wd);
  const BigParts P = big_parts(wd.bpart, nc);
  int bad = 0;
  if (nc > 0) {  // the pair kernel's CTAs looked at every atom
    for (int q = g.t; q < nc; q += g.G) bad |= P.bad[q];
  } else {
    for (int i = g.t; i < wd.natoms; i += g.G) {
      float4 p = x[i];
      bad |= (isfinite(p.x) && isfinite(p.y) && isfinite(p.z)) ? 0 : 1;
    }
  }
  if (grp_any<float>(g, fx, bad)) {
    if (g.t == 0) {
      head->bad = 1;
      head->dep = 0;
      head->flags = ABP_WFLAG_NONFINITE;
      atomicAdd(&ctr->nonfinite, 1);
    }
    return;
  }
  // COM distances on every warp, a dihedral on the last warp's last lane, the
  // CN's partial sums on the second warp
  __shared__ float part[kMaxCv][kBigThreads / 32][6][2];
  for (int k = 0; k < wd.g.d; ++k)
    if (wd.cv[k].type == ABP_CV_COM_DIST) big_com_part(g, wd.cv[k], x, part[k]);
  for (int k = 0; k < wd.g.d; ++k)
    if (wd.cv[k].type == ABP_CV_DIHEDRAL) cv_dihedral<float>(g, fx, k, x);
  if (kc >= 0 && g.warp == 1) {
    float h[1] = {0.f}, l[1] = {0.f};
    for (int q = g.lane; q < nc; q += 32) ff_add<float>(h[0], l[0], P.s[2 * q], P.s[2 * q + 1]);
    warp_sum_ff<1>(h, l);
    if (g.lane == 0) {
      fx->sh[kc] = h[0];
      fx->sl[kc] = l[0];
    }
  }
  g.sync();
  if (kc >= 0 && g.warp >= 2) {
    // A gradients: the CTAs' sums in chunk order, NQ components a thread (not needed before a5)
    float *jA = reinterpret_cast<float *>(js + big_layout(wd).jA);
    constexpr int NQ = 4;
    const int n3 = wd.cv[kc].na * 3, T = g.G - 64;
    for (int q0 = g.t - 64; q0 < n3; q0 += NQ * T) {
      float acc[NQ];
#pragma unroll
      for (int u = 0; u < NQ; ++u) acc[u] = 0.f;
#pragma unroll 9
      for (int w = 0; w < nc; ++w)
#pragma unroll
        for (int u = 0; u < NQ; ++u) {
          const int q = q0 + u * T;
          if (q < n3) acc[u] += P.g[(size_t)w * n3 + q];
        }
#pragma unroll
      for (int u = 0; u < NQ; ++u) {
        const int q = q0 + u * T;
        if (q < n3) jA[(q / 3) * 4 + q % 3] = acc[u];
      }
    }
  }
  if (g.warp == 0)
    for (int k = 0; k < wd.g.d; ++k)
      if (wd.cv[k].type == ABP_CV_COM_DIST) big_com_end(g, fx, k, x, part[k]);
  g.sync();
  const bool dep = (step % wd.stride) == 0;
  if (g.t < wd.g.d) axis_setup<float>(fx, g.t, dep);
  g.sync();
  if (dep && g.warp == 0) {
    // V_b(s_t) before this step's deposits: the FP64 shadow of a shared
    // grid, the value + compensation records of an own grid
    const GridDev &gd = wd.g;
    double acc = 0;
    if (g.lane < (1 << gd.d)) {
      double w = 1;
      long long node = 0, mul = 1;
      for (int k = 0; k < gd.d; ++k) {
        int hi = (g.lane >> k) & 1;
        double f = (double)fx->f[k];
        w *= hi ? f : 1.0 - f;
        node += mul * (hi ? fx->i1[k] : fx->i0[k]);
        mul *= gd.n[k];
      }
      double v;
      node = chk_node(gd, node);
      if (gd.shared) {
        v = gd.shadow[node * 4];
      } else {
        double vv[4];
        rec_values<double>(gd, reinterpret_cast<const unsigned char *>(gd.rec) + node * gd.rec_bytes, vv);
        v = vv[0];
      }
      acc = w * v;
    }
    for (int o = 1; o < 8; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (g.lane == 0) {
      double h = wd.w * exp(-acc * wd.inv_dT);
      head->h = h;
      head->hf = (float)h;
      if (log.rec) {
        unsigned long long slot = atomicAdd(log.count, 1ull);
        if (slot < log.cap) {
          abp_deposit_rec r;
          r.step = step;
          r.walker_id = wd.id;
          for (int k = 0; k < 3; ++k) {
            r.ic[k] = k < gd.d ? fx->ic_log[k] : 0;
            r.s[k] = k < gd.d ? (double)fx->sh[k] + (double)fx->sl[k] : 0.0;
          }
          r.height = h;
          log.rec[slot] = r;
        }
      }
    }
  }
  if (g.t == 0) {
    head->bad = 0;
    head->dep = dep ? 1 : 0;
    if (dep) fx->flags |= ABP_WFLAG_DEPOSIT;
    head->flags = fx->flags;
    for (int k = 0; k < kMaxCv; ++k) {
      head->sh[k] = fx->sh[k];
      head->sl[k] = fx->sl[k];
      head->da[k] = fx->da[k];
      head->dc[k] = fx->dc[k];
      head->df[k] = fx->df[k];
      head->ic_log[k] = fx->ic_log[k];
      for (int q = 0; q < 3; ++q) head->com_u[k][q] = fx->com_u[k][q];
      for (int a = 0; a < 4; ++a)
        for (int q = 0; q < 3; ++q) head->dih_g[k][a][q] = fx->dih_g[k][a][q];
    }
  }
  g.sync();
  if (look) big_lookup(g, fx, head, step);
}

// ---------------------------------------------------------------- deposit + refresh

// Stencil tables from the hill record (all CTAs of a walker build the same).
__device__ bool big_tables(const Grp &g, GroupFixed<float> *fx, const BigItem &it) {
  big_load_desc(g, fx, it.wd);
  const BigHead *head = reinterpret_cast<const BigHead *>(fx->wd.jscratch);
  if (!head->dep || head->bad) return false;
  if (g.t < kMaxCv) {
    fx->da[g.t] = head->da[g.t];
    fx->dc[g.t] = head->dc[g.t];
    fx->df[g.t] = head->df[g.t];
  }
  if (g.t == 0) fx->hf = head->hf;
  g.sync();
  build_tables<float>(g, fx);
  g.sync();
  return true;
}

__global__ void __launch_bounds__(kBigThreads) k_big_deposit(const BigItem *walkers) {
  extern __shared__ __align__(32) unsigned char smem[];
  Grp g = big_group();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  chain_wait();
  if (!big_tables(g, fx, walkers[blockIdx.x])) return;
  const WalkerDev &wd = fx->wd;
  const GridDev &gd = wd.g;
  const int d = gd.d;
  const int s0 = 2 * wd.R[0] + 1, s1 = d > 1 ? 2 * wd.R[1] + 1 : 1, s2 = d > 2 ? 2 * wd.R[2] + 1 : 1;
  const int total = s0 * s1 * s2;
  const int first = blockIdx.y * kStencilPerBlock, last = min(total, first + kStencilPerBlock);
  const long long n0 = gd.n[0], n01 = n0 * (d > 1 ? gd.n[1] : 1);
  const float h = fx->hf;
  for (int idx = first + g.t; idx < last; idx += g.G) {
    int o0 = idx % s0, r = idx / s0, o1 = r % s1, o2 = r / s1;
    int j0 = fx->tabJ[0][o0];
    int j1 = d > 1 ? fx->tabJ[1][o1] : 0;
    int j2 = d > 2 ? fx->tabJ[2][o2] : 0;
    if ((j0 | j1 | j2) < 0) continue;
    float G = h * fx->tabG[0][o0];
    if (d > 1) G = G * fx->tabG[1][o1];
    if (d > 2) G = G * fx->tabG[2][o2];
    float d0 = fx->tabD[0][o0], d1 = d > 1 ? fx->tabD[1][o1] : 0.f, d2 = d > 2 ? fx->tabD[2][o2] : 0.f;
    const long long node = chk_node(gd, j0 + n0 * j1 + n01 * j2);
    if (gd.shared) {
      double *p = gd.shadow + node * 4;
      atomicAdd(p, (double)G);
      atomicAdd(p + 1, (double)__fmul_rn(G, d0));
      if (d > 1) atomicAdd(p + 2, (double)__fmul_rn(G, d1));
      if (d > 2) atomicAdd(p + 3, (double)__fmul_rn(G, d2));
    } else {
      rmw_node<float>(gd, reinterpret_cast<unsigned char *>(gd.rec) + node * gd.rec_bytes, G, d0, d1, d2);
    }
  }
}

__global__ void __launch_bounds__(kBigThreads) k_big_refresh(const BigItem *walkers) {
  extern __shared__ __align__(32) unsigned char smem[];
  Grp g = big_group();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  chain_wait();
  if (!big_tables(g, fx, walkers[blockIdx.x])) return;
  const WalkerDev &wd = fx->wd;
  const GridDev &gd = wd.g;
  if (!gd.shared) return;
  const int d = gd.d;
  const int s0 = 2 * wd.R[0] + 1, s1 = d > 1 ? 2 * wd.R[1] + 1 : 1, s2 = d > 2 ? 2 * wd.R[2] + 1 : 1;
  const int total = s0 * s1 * s2;
  const int first = blockIdx.y * kStencilPerBlock, last = min(total, first + kStencilPerBlock);
  const long long n0 = gd.n[0], n01 = n0 * (d > 1 ? gd.n[1] : 1);
  for (int idx = first + g.t; idx < last; idx += g.G) {
    int o0 = idx % s0, r = idx / s0, o1 = r % s1, o2 = r / s1;
    int j0 = fx->tabJ[0][o0];
    int j1 = d > 1 ? fx->tabJ[1][o1] : 0;
    int j2 = d > 2 ? fx->tabJ[2][o2] : 0;
    if ((j0 | j1 | j2) < 0) continue;
    const long long node = chk_node(gd, j0 + n0 * j1 + n01 * j2);
    const double *p = gd.shadow + node * 4;
    float hi[4], lo[4];
    for (int q = 0; q < 4; ++q) {
      double v = q <= d ? p[q] : 0.0;
      hi[q] = (float)v;
      lo[q] = (float)(v - (double)hi[q]);
    }
    if (d == 1) {
      *reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(gd.rec) + node * 16) =
          make_float4(hi[0], hi[1], lo[0], lo[1]);
    } else {
      float4 *q = reinterpret_cast<float4 *>(reinterpret_cast<unsigned char *>(gd.rec) + node * 32);
      q[0] = make_float4(hi[0], hi[1], hi[2], hi[3]);
      q[1] = make_float4(lo[0], lo[1], lo[2], lo[3]);
    }
  }
}

// ---------------------------------------------------------------- a4 after deposits

// One warp per walker: the look-up after the step's deposits.
__global__ void __launch_bounds__(32) k_big_lookup(const BigItem *walkers, long long step) {
  extern __shared__ __align__(32) unsigned char smem[];
  const Grp g = big_group();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  big_load_desc(g, fx, walkers[blockIdx.x].wd);
  chain_wait();
  BigHead *head = reinterpret_cast<BigHead *>(fx->wd.jscratch);
  if (head->bad) return;
  if (g.t < kMaxCv) {
    fx->sh[g.t] = head->sh[g.t];
    fx->sl[g.t] = head->sl[g.t];
  }
  if (g.t == 0) fx->flags = head->flags;
  g.sync();
  if (g.t < fx->wd.g.d) axis_setup<float>(fx, g.t, false);
  g.sync();
  big_lookup(g, fx, head, step);
}

// ---------------------------------------------------------------- k_big_force

// a5 of one walker's atoms [blockIdx.x * kBigForceThreads, + kBigForceThreads):
// each thread sums its atom's terms in the walker's fixed order (CV by CV,
// list A before list B) and writes the walker's force buffer and, when given,
// the caller's. Closed loop (move): it then moves the atom, x += c1
// F_bias + c2 xi (this form takes no CV potential), the coordinates before
// the move to the trajectory records when given. A walker whose step saw
// non-finite coordinates gets no force and does not move.
__global__ void __launch_bounds__(kBigForceThreads) k_big_force(const BigItem *walkers, void *forces,
                                                                const long long *foff, long long force_step_off,
                                                                int mode, long long step, MdParams md, int move,
                                                                void *xio, const long long *coff, void *traj,
                                                                const long long *toff, long long traj_step_off) {
  const BigItem it = walkers[blockIdx.y];
  const WalkerDev &wd = *it.wd;
  const int i = blockIdx.x * kBigForceThreads + threadIdx.x;
  float n[3] = {0.f, 0.f, 0.f};
  if (move && i < wd.natoms) md_normals(md.seed, it.stream, step, i, n);  // needs no earlier result
  chain_wait();
  if (i >= wd.natoms) return;
  unsigned char *js = reinterpret_cast<unsigned char *>(wd.jscratch);
  const BigHead *head = reinterpret_cast<const BigHead *>(js);
  float4 *fb = reinterpret_cast<float4 *>(wd.fbuf);
  float4 *fo = forces ? reinterpret_cast<float4 *>(forces) + foff[it.widx] + force_step_off : fb;
  const int fmode = forces ? mode : ABP_FORCES_OVERWRITE;
  if (head->bad) {
    if (fmode == ABP_FORCES_OVERWRITE) fo[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i == 0) wd.state->flags = ABP_WFLAG_NONFINITE;
    return;
  }
  const BigLayout L = big_layout(wd);
  const int32_t *tt = reinterpret_cast<const int32_t *>(js + L.terms) + (size_t)i * kAtomTerms;
  const int ne = js[L.nterm + i];
  const float4 *jA = reinterpret_cast<const float4 *>(js + L.jA);
  const float4 *jB = reinterpret_cast<const float4 *>(js + L.jB);
  float f0 = 0.f, f1 = 0.f, f2 = 0.f;
  for (int q = 0; q < ne; ++q) {
    const int code = tt[q], kind = code & 7, k = (code >> 3) & 3, pos = code >> 5;
    const float dv = head->dv[k];
    if (kind == kTermComA || kind == kTermComB) {
      const float ux = head->com_u[k][0] * dv, uy = head->com_u[k][1] * dv, uz = head->com_u[k][2] * dv;
      if (kind == kTermComA) {
        const float w = wd.cv[k].wa[pos];
        f0 += w * ux;
        f1 += w * uy;
        f2 += w * uz;
      } else {
        const float w = wd.cv[k].wb[pos];
        f0 -= w * ux;
        f1 -= w * uy;
        f2 -= w * uz;
      }
    } else if (kind == kTermDih) {
      f0 -= dv * head->dih_g[k][pos][0];
      f1 -= dv * head->dih_g[k][pos][1];
      f2 -= dv * head->dih_g[k][pos][2];
    } else {
      const float4 j = kind == kTermCnA ? jA[pos] : jB[pos];
      f0 -= dv * j.x;
      f1 -= dv * j.y;
      f2 -= dv * j.z;
    }
  }
  fb[i] = make_float4(f0, f1, f2, 0.f);
  if (fo != fb) {
    if (fmode == ABP_FORCES_ACCUMULATE) {
      float4 o = fo[i];
      o.x += f0;
      o.y += f1;
      o.z += f2;
      fo[i] = o;
    } else {
      fo[i] = make_float4(f0, f1, f2, 0.f);
    }
  }
  if (move) {
    float4 *x = reinterpret_cast<float4 *>(xio) + coff[it.widx] + i;
    float4 p = *x;
    if (traj) reinterpret_cast<float4 *>(traj)[toff[it.widx] + traj_step_off + i] = p;
    const float c1 = (float)md.c1, c2 = (float)md.c2;
    p.x += c1 * f0 + c2 * n[0];
    p.y += c1 * f1 + c2 * n[1];
    p.z += c1 * f2 + c2 * n[2];
    *x = p;
  }
}

// ---------------------------------------------------------------- launcher

cudaError_t launch_big_step(const BigArgs &a, cudaStream_t st) {
  const size_t fixed = (size_t)fixed_bytes_f();
  // all phases: without a deposit this step the grid does not change, and the
  // look-up goes with the CVs
  const bool look = !a.phases && !a.any_deposit;
  const int ph = a.phases ? a.phases : a.any_deposit ? 31 : 19;
  LaunchTimer *tm = a.timer;
  auto t0 = [&](const char *k) {
    nvtxRangePushA(k);
    if (tm) tm->begin(k, st);
  };
  auto t1 = [&](const char *k) {
    if (tm) tm->end(k, st);
    nvtxRangePop();
  };
  cudaError_t e = cudaSuccess;
  if ((ph & 1) && a.ncn_items > 0) {
    e = smem_attr(reinterpret_cast<const void *>(k_big_cn), a.cn_smem);
    if (e != cudaSuccess) return e;
    t0("k_big_cn");
    e = launch_chained(k_big_cn, a.ncn_items, kBigCnThreads, a.cn_smem, st, a.cn_items, a.coords, a.coff, a.step_off);
    if (e != cudaSuccess) return e;
    t1("k_big_cn");
  }
  if (ph & 2) {
    t0("k_big_cvs");
    e = launch_chained(k_big_cvs, a.nw, kBigThreads, fixed, st, a.walkers, a.coords, a.coff, a.step_off, a.step, a.log,
                       a.ctr, look ? 1 : 0);
    if (e != cudaSuccess) return e;
    t1("k_big_cvs");
  }
  dim3 grid(a.nw, (a.max_stencil + kStencilPerBlock - 1) / kStencilPerBlock);
  if (ph & 4) {
    t0("k_big_deposit");
    e = launch_chained(k_big_deposit, grid, kBigThreads, fixed, st, a.walkers);
    if (e != cudaSuccess) return e;
    t1("k_big_deposit");
  }
  if ((ph & 8) && a.any_shared) {
    t0("k_big_refresh");
    e = launch_chained(k_big_refresh, grid, kBigThreads, fixed, st, a.walkers);
    if (e != cudaSuccess) return e;
    t1("k_big_refresh");
  }
  if ((ph & 16) && !look) {
    t0("k_big_lookup");
    e = launch_chained(k_big_lookup, a.nw, 32, fixed, st, a.walkers, a.step);
    if (e != cudaSuccess) return e;
    t1("k_big_lookup");
  }
  if (ph & 16) {
    t0("k_big_force");
    const MdParams md = a.md ? *a.md : MdParams{};
    e = launch_chained(k_big_force, dim3((a.max_atoms + kBigForceThreads - 1) / kBigForceThreads, a.nw),
                       kBigForceThreads, 0, st, a.walkers, a.forces, a.foff, a.force_step_off, a.mode, a.step, md,
                       a.md ? 1 : 0, a.xio, a.coff, a.traj, a.toff, a.traj_step_off);
    if (e != cudaSuccess) return e;
    t1("k_big_force");
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------- hill records

// One CTA per (record, block of stencil nodes): the record's axis state from
// its centre, its tables, and a plain FP64 read-modify-write of the shadow
// (records of one launch have disjoint boxes), or the FP32 refresh.
__global__ void __launch_bounds__(kBigThreads) k_apply_hills(const WalkerDev *shape, const HillDev *recs, int refresh) {
  extern __shared__ __align__(32) unsigned char smem[];
  Grp g = big_group();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  const int *src = reinterpret_cast<const int *>(shape);
  int *dst = reinterpret_cast<int *>(&fx->wd);
  for (int i = g.t; i < (int)(sizeof(WalkerDev) / 4); i += g.G) dst[i] = src[i];
  const HillDev r = recs[blockIdx.x];
  if (g.t == 0) {
    fx->clamped = 0;
    fx->flags = 0;
  }
  g.sync();
  const GridDev &gd = fx->wd.g;
  if (g.t < kMaxCv) {
    float h = (float)r.s[g.t];
    fx->sh[g.t] = h;
    fx->sl[g.t] = (float)(r.s[g.t] - (double)h);
  }
  g.sync();
  if (g.t < gd.d) axis_setup<float>(fx, g.t, true);
  g.sync();
  build_tables<float>(g, fx);
  g.sync();
  const WalkerDev &wd = fx->wd;
  const int d = gd.d;
  const int s0 = 2 * wd.R[0] + 1, s1 = d > 1 ? 2 * wd.R[1] + 1 : 1, s2 = d > 2 ? 2 * wd.R[2] + 1 : 1;
  const int total = s0 * s1 * s2;
  const int first = blockIdx.y * kStencilPerBlock, last = min(total, first + kStencilPerBlock);
  const long long n0 = gd.n[0], n01 = n0 * (d > 1 ? gd.n[1] : 1);
  const float hf = (float)r.h;
  for (int idx = first + g.t; idx < last; idx += g.G) {
    int o0 = idx % s0, rr = idx / s0, o1 = rr % s1, o2 = rr / s1;
    int j0 = fx->tabJ[0][o0];
    int j1 = d > 1 ? fx->tabJ[1][o1] : 0;
    int j2 = d > 2 ? fx->tabJ[2][o2] : 0;
    if ((j0 | j1 | j2) < 0) continue;
    const long long node = chk_node(gd, j0 + n0 * j1 + n01 * j2);
    double *p = gd.shadow + node * 4;
    if (!refresh) {
      float G = hf * fx->tabG[0][o0];
      if (d > 1) G = G * fx->tabG[1][o1];
      if (d > 2) G = G * fx->tabG[2][o2];
      p[0] += (double)G;
      p[1] += (double)__fmul_rn(G, fx->tabD[0][o0]);
      if (d > 1) p[2] += (double)__fmul_rn(G, fx->tabD[1][o1]);
      if (d > 2) p[3] += (double)__fmul_rn(G, fx->tabD[2][o2]);
    } else {
      float hi[4], lo[4];
      for (int q = 0; q < 4; ++q) {
        double v = q <= d ? p[q] : 0.0;
        hi[q] = (float)v;
        lo[q] = (float)(v - (double)hi[q]);
      }
      unsigned char *rec = reinterpret_cast<unsigned char *>(gd.rec) + node * gd.rec_bytes;
      if (d == 1) {
        *reinterpret_cast<float4 *>(rec) = make_float4(hi[0], hi[1], lo[0], lo[1]);
      } else {
        float4 *q = reinterpret_cast<float4 *>(rec);
        q[0] = make_float4(hi[0], hi[1], hi[2], hi[3]);
        q[1] = make_float4(lo[0], lo[1], lo[2], lo[3]);
      }
    }
  }
}

cudaError_t launch_apply_hills(const WalkerDev *shape, const HillDev *recs, int n, int max_stencil, bool refresh,
                               cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  dim3 grid(n, (max_stencil + kStencilPerBlock - 1) / kStencilPerBlock);
  k_apply_hills<<<grid, kBigThreads, fixed_bytes_f(), st>>>(shape, recs, refresh ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t read_hill_heads(const WalkerDev *const *wd_host, int n, double *s3h, int *dep, cudaStream_t st) {
  // wd_host[i] is a host copy of walker i's descriptor (for its jscratch)
  cudaError_t e = cudaStreamSynchronize(st);
  for (int i = 0; i < n && e == cudaSuccess; ++i) {
    BigHead head;
    e = cudaMemcpy(&head, wd_host[i]->jscratch, sizeof head, cudaMemcpyDeviceToHost);
    for (int k = 0; k < 3; ++k) s3h[4 * i + k] = (double)head.sh[k] + (double)head.sl[k];
    s3h[4 * i + 3] = head.h;
    dep[i] = head.dep && !head.bad;
  }
  return e;
}

// The phased form takes coordination numbers of up to kBigMaxA A atoms (200 KB
// at 16 + 8 x 12 bytes an atom, the shared memory of a pair CTA of eight
// warps; the CTAs of two warps stay below that).
constexpr int kBigMaxA = 200 * 1024 / (16 + 8 * 12);
bool big_cn_too_large(const WalkerDev &hd) {
  const int k = big_cn_index(hd);
  return k >= 0 && hd.cv[k].na > kBigMaxA;
}

size_t big_cn_smem(const WalkerDev &hd) {
  int k = big_cn_index(hd);
  if (k < 0) return 0;
  return (size_t)hd.cv[k].na * 16 + (size_t)(kBigCnThreads / 32) * hd.cv[k].na * 12;
}

}  // namespace abp
