// abp_split.cu -- the split form of the open-loop force call (abp_run,
// abp_step): a call over recorded coordinates in three launches per block of
// steps instead of one group per walker stepping through them.
//
// Only the grid ties a walker's steps together: a step's CVs and Jacobian
// factors depend on its coordinates alone, and its forces on those and on
// dV_b/ds. So
//
//   k_sp_cv     a1 of (walker, window of steps) items: walkers whose CVs one
//               thread evaluates (COM distances, dihedrals, small RMSDs)
//   k_sp_cn     a1 of (walker, steps) items: the other FP32 walkers
//               (coordination numbers, long atom lists), a warp or a CTA per
//               step
//   k_sp_chain  a2 .. a4, one CTA per well-tempered walker: the steps between
//               two deposits interpolate side by side, the deposits in order
//   k_sp_hist   a3 + a4 of mABP walkers: hills of a fixed height on the
//               nearest node do not depend on look-ups, so a walker's grid is
//               cut into slices of its last axis, one CTA each, without any
//               exchange between them
//   k_sp_force  a5 of (walker, steps) items from the step records
//   k_sp_cnf    the same from the coordination numbers' gradient records
//
// run over step records (StepRec) kept in a scratch block of the call, so the
// parts without a chain use the whole chip however few walkers there are. The
// arithmetic per step is the windowed form's (abp_window_ops.cuh), and a
// coordination number's sum that of a group of 128 threads: the same bits as
// the forms with a group per walker at their default width. FP32 grids.
//
// One group per walker against this form (GB300, whole calls): 3 walkers x 101
// steps, 53 x 307 pairs, 4.04 ms -> 41 us; 1000 walkers x 25 steps, 40 x 400
// pairs, 2.04 ms -> 0.59 ms; 64 walkers x 1000 steps of recorded frames 218
// -> 154 us; two RMSDs with a 441-node hill every step 1.01 ms -> 176 us.
#include <cuda_runtime.h>

#include "abp_device.cuh"
#include "abp_launch.h"
#include "abp_window_ops.cuh"

namespace abp {

namespace {

using Step = StepRec<float>;
constexpr int kStepWords = (int)(sizeof(Step) / 4);
constexpr int kCvThreads = 128, kCnThreads = 128, kChainThreads = 512, kHistThreads = 128, kForceThreads = 128,
              kShortThreads = 256, kOneThreads = (4 + 2) * 32;
constexpr int kHistWin = 64;  // most mABP hills applied to a node between its load and its store

__host__ __device__ constexpr int fixed_bytes_f() { return (int)((sizeof(GroupFixed<float>) + 31) & ~(size_t)31); }
__host__ __device__ constexpr int up32(int x) { return (x + 31) & ~31; }

__device__ __forceinline__ Grp cta_grp() {
  Grp g;
  g.G = blockDim.x;
  g.gid = 0;
  g.t = threadIdx.x;
  g.lane = threadIdx.x & 31;
  g.warp = threadIdx.x >> 5;
  g.nwarps = blockDim.x >> 5;
  return g;
}

__device__ __forceinline__ void load_words(const Grp &g, void *dst, const void *src, int words) {
  const int *s = reinterpret_cast<const int *>(src);
  int *d = reinterpret_cast<int *>(dst);
  for (int i = g.t; i < words; i += g.G) d[i] = s[i];
}

__device__ __forceinline__ Step *walker_steps_of(const SplitArgs &a, int slot) {
  return reinterpret_cast<Step *>(a.recs) + (size_t)slot * a.nsteps;
}

// The CV lists (and COM weights) of a walker into shared memory. Caller syncs.
__device__ void stage_lists(const Grp &g, const WalkerDev &wd, unsigned char *mem, const int32_t **ia,
                            const int32_t **ib, const float **wa, const float **wb) {
  unsigned char *cur = mem;
  for (int k = 0; k < wd.g.d; ++k) {
    const CvDev &c = wd.cv[k];
    int32_t *la = reinterpret_cast<int32_t *>(cur), *lb = la + c.na;
    for (int i = g.t; i < c.na; i += g.G) la[i] = c.ia[i];
    for (int i = g.t; i < c.nb; i += g.G) lb[i] = c.ib[i];
    cur += align16((c.na + c.nb) * 4);
    float *pa = reinterpret_cast<float *>(cur), *pb = pa + c.na;
    if (c.type == ABP_CV_COM_DIST) {
      for (int i = g.t; i < c.na; i += g.G) pa[i] = c.wa[i];
      for (int i = g.t; i < c.nb; i += g.G) pb[i] = c.wb[i];
      cur += align16((c.na + c.nb) * 4);
    }
    if (g.t == 0) {
      ia[k] = la;
      ib[k] = lb;
      wa[k] = pa;
      wb[k] = pb;
    }
  }
}

__host__ __device__ inline int list_bytes(const CvDev *cv, int d) {
  int b = 0;
  for (int k = 0; k < d; ++k) {
    b += align16((cv[k].na + cv[k].nb) * 4);
    if (cv[k].type == ABP_CV_COM_DIST) b += align16((cv[k].na + cv[k].nb) * 4);
  }
  return up32(b);
}

// ---------------------------------------------------------------- a1, windows

// Shared memory of k_sp_cv: GroupFixed | W step records | lists | W rows.
struct CvLayout {
  int recs, lists, xs, xst, total;
};
__host__ __device__ inline CvLayout cv_layout(int natoms, const CvDev *cv, int d, int W) {
  CvLayout L;
  L.recs = fixed_bytes_f();
  L.lists = up32(L.recs + W * (int)sizeof(Step));
  L.xs = L.lists + list_bytes(cv, d);
  L.xst = natoms | 1;  // an odd row stride: one row per thread without bank conflicts
  L.total = L.xs + W * L.xst * 16;
  return L;
}

// The step records of nt steps whose coordinates are on their way to xs (rows
// of xst records) and whose lists are being staged: one lane per (CV, step),
// two for a COM distance, the finiteness of every atom, the flags.
__device__ __forceinline__ void window_records(const Grp &g, GroupFixed<float> *fx, const float4 *xs, int xst, Step *st,
                                               int nt, long long s0, DevCounters *ctr) {
  const WalkerDev &wd = fx->wd;
  const int d = wd.g.d, natoms = wd.natoms;
  if (g.t == 0) fx->winbad[0] = 0;
  cp_async_wait_all();
  __syncthreads();
  // tasks: whole warps per CV; warps go round the task list
  int base[kMaxCv + 1];
  base[0] = 0;
  for (int k = 0; k < d; ++k) base[k + 1] = base[k] + align32((wd.cv[k].type == ABP_CV_COM_DIST ? 2 : 1) * nt);
  for (int task = g.t; task < base[d]; task += g.G) {
    int k = 0;
    while (k + 1 < d && task >= base[k + 1]) ++k;
    const int r = task - base[k];
    if (wd.cv[k].type == ABP_CV_COM_DIST) {
      const int j = min(r >> 1, nt - 1);
      window_com2<float>(fx, xs + j * xst, k, (s0 + j) % wd.stride == 0, (r >> 1) < nt, r & 1, st[j]);
    } else if (r < nt) {
      window_cv<float>(fx, xs + r * xst, k, (s0 + r) % wd.stride == 0, st[r]);
    }
  }
  unsigned mine = 0;
  for (Iter2 it(g.t, g.G, natoms); it.j < nt; it.next())
    if (!finite_rec<float>(xs[it.j * xst + it.i])) mine |= 1u << it.j;
  mine = __reduce_or_sync(0xffffffffu, mine);
  if (g.lane == 0 && mine) atomicOr(&fx->winbad[0], mine);
  __syncthreads();
  const unsigned bad = fx->winbad[0];
  if (g.t == 0 && bad) atomicAdd(&ctr->nonfinite, __popc(bad));
  for (int j = g.t; j < nt; j += g.G) {
    if ((bad >> j) & 1)
      st[j].flags = ABP_WFLAG_NONFINITE;
    else
      step_flags<float>(d, (s0 + j) % wd.stride == 0, st[j]);
  }
  __syncthreads();
}

// One window (W steps, as window_steps gives for the walker) of one walker:
// its coordinates into shared memory, one lane per (CV, step) -- two for a
// COM distance --, the finiteness of every atom on the threads left over,
// the records out in one coalesced copy.
__global__ void __launch_bounds__(kCvThreads) k_sp_cv(SplitArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  const Grp g = cta_grp();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  const TableEntry te = a.table[blockIdx.x];
  load_words(g, &fx->wd, te.wd, (int)(sizeof(WalkerDev) / 4));
  __syncthreads();
  const WalkerDev &wd = fx->wd;
  const int d = wd.g.d, natoms = wd.natoms, W = window_steps(natoms, wd.cv, d, 16);
  const int t0 = blockIdx.y * W, nt = min(W, a.nsteps - t0);
  if (nt <= 0) return;
  const CvLayout L = cv_layout(natoms, wd.cv, d, W);
  Step *st = reinterpret_cast<Step *>(smem + L.recs);
  float4 *xs = reinterpret_cast<float4 *>(smem + L.xs);
  const float4 *cin = reinterpret_cast<const float4 *>(a.coords) + a.coff[te.idx] + (a.t0 + t0) * a.cstride;
  for (Iter2 it(g.t, g.G, natoms); it.j < nt; it.next())
    cp_async16(xs + it.j * L.xst + it.i, cin + (long long)it.j * a.cstride + it.i);
  cp_async_commit();
  stage_lists(g, wd, smem + L.lists, fx->ia, fx->ib, fx->wa, fx->wb);
  window_records(g, fx, xs, L.xst, st, nt, a.step0 + a.t0 + t0, a.ctr);
  load_words(g, walker_steps_of(a, blockIdx.x) + t0, st, nt * kStepWords);
}

// ---------------------------------------------------------------- a1 with coordination numbers

constexpr int kCnWarps = kCnThreads / 32;
constexpr int kCnBatch = 8;  // most consecutive steps of a warp in k_sp_cn

constexpr int kCnStage = 10 * 1024;  // most bytes of a step's coordinates that k_sp_cn stages per warp

// Shared memory of k_sp_cn: the CTA's step records, per warp its A gradients,
// then (walkers of at most kCnStage bytes of atoms) the coordinates of each
// warp's step.
__host__ __device__ inline int cn_recs_bytes() { return up32(kCnWarps * kCnBatch * (int)sizeof(Step)); }
__host__ __device__ inline int cn_lig_floats(const CvDev *cv, int d) {
  int na = 0;
  for (int k = 0; k < d; ++k)
    if (cv[k].type == ABP_CV_COORD && cv[k].na > na) na = cv[k].na;
  return na * 3;
}
__host__ __device__ inline int cn_stage_offset(const CvDev *cv, int d) {
  return cn_recs_bytes() + up32(kCnWarps * cn_lig_floats(cv, d) * 4);
}
__host__ __device__ inline int cn_bytes(const CvDev *cv, int d, int natoms) {
  return cn_stage_offset(cv, d) + (natoms * 16 <= kCnStage ? kCnWarps * natoms * 16 : 0);
}

// Gradient records of one step: per COORD CV, list A then list B.
__host__ __device__ inline int cn_records(const CvDev *cv, int d) {
  int n = 0;
  for (int k = 0; k < d; ++k)
    if (cv[k].type == ABP_CV_COORD) n += cv[k].na + cv[k].nb;
  return n;
}

// Every coordinate of the step finite? (0 x is NaN for an infinite or NaN x.)
__device__ __forceinline__ bool step_finite(const float4 *x, int natoms, int t, int T) {
  float z = 0.f;
  for (int i = t; i < natoms; i += T) {
    const float4 p = x[i];
    z = __fmaf_rn(p.x, 0.f, __fmaf_rn(p.y, 0.f, __fmaf_rn(p.z, 0.f, z)));
  }
  return z == 0.f;
}

// The records of nt steps (their CVs' values, Jacobian factors and flags in
// place, the dihedrals not) finished by one warp: dihedrals one step a lane,
// the axis states one (step, CV) a lane, flags, the copy out.
__device__ __forceinline__ void finish_records(const WalkerDev &wd, Step *st, int nt, unsigned bad, long long s0,
                                               const float4 *x, long long cstride, int lane, Step *out) {
  const int d = wd.g.d;
  for (int k = 0; k < d; ++k)
    if (wd.cv[k].type == ABP_CV_DIHEDRAL && lane < nt && !((bad >> lane) & 1)) {
      float phi, lo;
      Step &s = st[lane];
      s.cfl[k] = dihedral_eval<float>(wd.cv[k], wd.cv[k].ia, x + lane * cstride, phi,
                                      reinterpret_cast<float(*)[3]>(s.jac[k]), lo);
      s.s[k] = phi;
      s.sl[k] = lo;
    }
  __syncwarp();
  for (int i = lane; i < nt * d; i += 32) {
    const int j = i / d, k = i - j * d;
    if (!((bad >> j) & 1))
      window_cv_rec<float>(wd, k, st[j].s[k], st[j].sl[k], st[j].cfl[k], (s0 + j) % wd.stride == 0, st[j]);
  }
  __syncwarp();
  if (lane < nt) {
    if ((bad >> lane) & 1)
      st[lane].flags = ABP_WFLAG_NONFINITE;
    else
      step_flags<float>(d, (s0 + lane) % wd.stride == 0, st[lane]);
  }
  __syncwarp();
  const int *src = reinterpret_cast<const int *>(st);
  int *dst = reinterpret_cast<int *>(out);
  for (int i = lane; i < nt * kStepWords; i += 32) dst[i] = src[i];
}

// Steps of one walker, all CVs. A coordination number is summed as four
// warps' parts (B-groups 8 v .. 8 v + 7 of 32, v = 0 .. 3) that meet in order:
// PER_WARP, the four are taken one after another by the warp that has the
// step (a.chunk steps a warp, no barrier anywhere: the form for batches that
// fill the chip); otherwise by the CTA's four warps, one step a CTA. The same
// sums, so the same bits. STAGED: a step's atoms are copied to shared memory
// first (all in flight at once, the next step's asked into L2 meanwhile);
// else they are read where they lie. LONG: a coordination number of the batch
// has more than 40 A atoms. 1000 walkers x 25 steps of 40 x 400 pairs, whole
// calls: 587 us staged without LONG, 611 with its path in the code, 614 not
// staged. ~120 registers a thread: four CTAs an SM.
template <bool PER_WARP, bool STAGED, bool LONG>
__global__ void __launch_bounds__(kCnThreads, 4) k_sp_cn(SplitArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  __shared__ float red[kCnWarps][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int me = PER_WARP ? lane : (int)threadIdx.x, team = PER_WARP ? 32 : kCnThreads;
  const TableEntry te = a.table[blockIdx.x];
  const WalkerDev &wd = *te.wd;
  const int d = wd.g.d, natoms = wd.natoms;
  const int tb = PER_WARP ? (blockIdx.y * kCnWarps + warp) * a.chunk : blockIdx.y;
  const int nt = min(PER_WARP ? a.chunk : 1, a.nsteps - tb);
  if (nt <= 0) return;
  Step *st = reinterpret_cast<Step *>(smem) + (PER_WARP ? warp * kCnBatch : 0);
  float *ligs = reinterpret_cast<float *>(smem + cn_recs_bytes());
  const int nlig = cn_lig_floats(wd.cv, d);
  float4 *buf = reinterpret_cast<float4 *>(smem + cn_stage_offset(wd.cv, d)) + (PER_WARP ? warp * natoms : 0);
  const float4 *cin = reinterpret_cast<const float4 *>(a.coords) + a.coff[te.idx] + (a.t0 + tb) * a.cstride;
  const long long s0 = a.step0 + a.t0 + tb;
  unsigned bad = 0;
  for (int j = 0; j < nt; ++j) {
    const float4 *xg = cin + j * a.cstride;
    if (STAGED) {
      for (int i = me; i < natoms; i += team) cp_async16(buf + i, xg + i);
      cp_async_commit();
      if (j + 1 < nt)
        for (int i = me * 8; i < natoms; i += team * 8)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(xg + a.cstride + i));
      cp_async_wait_all();
      if (PER_WARP)
        __syncwarp();
      else
        __syncthreads();
    }
    const float4 *x = STAGED ? buf : xg;
    const bool fin = step_finite(x, natoms, me, team);
    if (PER_WARP ? __any_sync(0xffffffffu, !fin) : __syncthreads_or(!fin)) {
      bad |= 1u << j;
      continue;
    }
    float4 *J = reinterpret_cast<float4 *>(a.jac) + ((size_t)blockIdx.x * a.nsteps + tb + j) * a.jstride;
    for (int k = 0; k < d; ++k) {
      const CvDev &c = wd.cv[k];
      if (c.type == ABP_CV_COM_DIST) {
        if (PER_WARP || warp == 0) {
          float s = 0.f, sl = 0.f;
          const int fl = com_one_warp(c, c.ia, c.ib, c.wa, c.wb, x, lane, s, sl, st[j].jac[k]);
          if (lane == 0) {
            st[j].s[k] = s;
            st[j].sl[k] = sl;
            st[j].cfl[k] = fl;
          }
        }
      } else if (c.type == ABP_CV_COORD) {
        const float c6 = -6.f * (float)c.inv_r0sq;
        float4 *jA = J, *jB = J + c.na;
        J += c.na + c.nb;
        float sh, sl;
        if (PER_WARP) {
          float *lig = ligs + warp * nlig;
          float h[kCnWarps], l[kCnWarps];
#pragma unroll 1
          for (int v = 0; v < kCnWarps; ++v) {
            float ph, pl;
            cn_warp_any<LONG>(c, c.ia, c.ib, x, jB, lig, v > 0, lane, 8 * v, 8 * kCnWarps, ph, pl);
#pragma unroll
            for (int q = 0; q < kCnWarps; ++q)
              if (q == v) {
                h[q] = ph;
                l[q] = pl;
              }
          }
          warp_sum_ff<kCnWarps>(h, l);
          sh = h[0];
          sl = l[0];
#pragma unroll
          for (int v = 1; v < kCnWarps; ++v) ff_add<float>(sh, sl, h[v], l[v]);
          __syncwarp();
          for (int i = lane; i < c.na; i += 32)
            jA[i] = make_float4(__fmul_rn(c6, lig[3 * i]), __fmul_rn(c6, lig[3 * i + 1]),
                                __fmul_rn(c6, lig[3 * i + 2]), 0.f);
          __syncwarp();
        } else {
          float h[1], l[1];
          cn_warp_any<LONG>(c, c.ia, c.ib, x, jB, ligs + warp * c.na * 3, false, lane, 8 * warp, 8 * kCnWarps, h[0], l[0]);
          warp_sum_ff<1>(h, l);
          if (lane == 0) {
            red[warp][0] = h[0];
            red[warp][1] = l[0];
          }
          __syncthreads();
          sh = red[0][0];
          sl = red[0][1];
#pragma unroll
          for (int v = 1; v < kCnWarps; ++v) ff_add<float>(sh, sl, red[v][0], red[v][1]);
          for (int i = threadIdx.x; i < c.na; i += kCnThreads) {
            float s3[3];
#pragma unroll
            for (int e = 0; e < 3; ++e) {
              s3[e] = ligs[3 * i + e];
#pragma unroll
              for (int v = 1; v < kCnWarps; ++v) s3[e] = __fadd_rn(s3[e], ligs[(v * c.na + i) * 3 + e]);
            }
            jA[i] = make_float4(__fmul_rn(c6, s3[0]), __fmul_rn(c6, s3[1]), __fmul_rn(c6, s3[2]), 0.f);
          }
          __syncthreads();  // the scratch is free again
        }
        if (PER_WARP ? lane == 0 : threadIdx.x == 0) {
          st[j].s[k] = sh;
          st[j].sl[k] = sl;
          st[j].cfl[k] = 0;
        }
      }
    }
    if (STAGED && PER_WARP) __syncwarp();  // every lane is done with the buffer
  }
  if (PER_WARP)
    __syncwarp();
  else
    __syncthreads();
  if (PER_WARP || warp == 0) {
    if (lane == 0 && bad) atomicAdd(&a.ctr->nonfinite, __popc(bad));
    finish_records(wd, st, nt, bad, s0, cin, a.cstride, lane, walker_steps_of(a, blockIdx.x) + tb);
  }
}

// The list entries an atom appears in, for a5 of walkers with gradient
// records: per atom their count and [slot][atom] pairs of a code, kind | k <<
// 2, and what the kind needs: a COM weight (list B's negated) as bits, or the
// record's position. List by list (an atom appears at most once in a list),
// which is the terms' order: CV by CV, list A before list B. One group per
// walker.
enum { kCom = 0, kDih = 1, kCn = 2 };

__device__ __forceinline__ int2 *atom_terms_of(const SplitArgs &a, int slot) {
  return reinterpret_cast<int2 *>(a.terms) + (size_t)slot * a.term_stride;
}
__device__ __forceinline__ int *atom_counts_of(const SplitArgs &a, int slot, int natoms) {
  return reinterpret_cast<int *>(atom_terms_of(a, slot) + (size_t)natoms * kAtomTerms);
}

__device__ void list_atom_terms(const Grp &g, const WalkerDev &wd, int2 *terms, int *cnt) {
  const int natoms = wd.natoms, d = wd.g.d;
  for (int i = g.t; i < natoms; i += g.G) cnt[i] = 0;
  int jpos = 0;
  for (int k = 0; k < d; ++k) {
    const CvDev &c = wd.cv[k];
    const bool com = c.type == ABP_CV_COM_DIST, cn = c.type == ABP_CV_COORD;
    for (int l = 0; l < (com || cn ? 2 : 1); ++l) {
      const int n = l ? c.nb : (com || cn ? c.na : 4);
      const int32_t *list = l ? c.ib : c.ia;
      g.sync();
      for (int i = g.t; i < n; i += g.G) {
        const int at = list[i], slot = cnt[at];
        const int arg = com ? __float_as_int(l ? -c.wb[i] : c.wa[i]) : cn ? jpos + (l ? c.na : 0) + i : i;
        terms[slot * natoms + at] = make_int2((com ? kCom : cn ? kCn : kDih) | (k << 2), arg);
        cnt[at] = slot + 1;
      }
    }
    if (cn) jpos += c.na + c.nb;
  }
  g.sync();
}

// a4 of one step from its record, V and dV/ds back into it (the arithmetic of
// interp_one; the Jacobian factors are scaled where a5 reads them).
template <int DIM>
__device__ __forceinline__ void step_lookup(const WalkerDev &wd, Step *sp) {
  if (sp->flags & ABP_WFLAG_NONFINITE) return;
  Step s;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    s.i0[k] = sp->i0[k];
    s.i1[k] = sp->i1[k];
    s.f[k] = sp->f[k];
    s.s[k] = sp->s[k];
  }
  const int clamped = sp->clamped;
  float4 ca[1 << DIM], cb[1 << DIM];
  interp_load<float, DIM>(wd, s, ca, cb);
  float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int c = 0; c < (1 << DIM); ++c) {
    const float wc = corner_weight<float, DIM>(s, c);
    float v[4];
    rec_vals<float, DIM>(ca[c], cb[c], v);
#pragma unroll
    for (int q = 0; q <= DIM; ++q) acc[q] = fma_rn(wc, v[q], acc[q]);
  }
  if (wd.method == ABP_METHOD_MABP) {  // the nearest node's histograms
    float V, dvm[3] = {0.f, 0.f, 0.f};
    mabp_bias<float>(wd, acc, V, dvm);
    acc[0] = V;
#pragma unroll
    for (int k = 0; k < DIM; ++k) acc[1 + k] = dvm[k];
  }
  sp->V = acc[0];
#pragma unroll
  for (int k = 0; k < DIM; ++k)
    sp->dv[k] = add_rn(((clamped >> k) & 1) ? 0.f : acc[1 + k], wall_grad<float>(wd, k, s.s[k], sp->sl[k]));
}

// The walker's state after the call's last step.
__device__ __forceinline__ void state_out(const WalkerDev &wd, const Step &s, long long step) {
  if (s.flags & ABP_WFLAG_NONFINITE) {
    wd.state->flags = ABP_WFLAG_NONFINITE;
    return;
  }
  WalkerState ws;
  for (int k = 0; k < 3; ++k) {
    ws.s[k] = k < wd.g.d ? (double)s.s[k] + (double)s.sl[k] : 0.0;
    ws.dV[k] = k < wd.g.d ? (double)s.dv[k] : 0.0;
  }
  ws.V = (double)s.V;
  ws.flags = s.flags;
  ws.pad = 0;
  ws.step = step;
  *wd.state = ws;
}

// The group of one warp of g (its reductions and loops; no group barrier).
__device__ __forceinline__ Grp warp_grp(const Grp &g) {
  Grp w = g;
  w.G = 32;
  w.t = g.lane;
  w.warp = 0;
  w.nwarps = 1;
  return w;
}

// a2 of a deposit by one warp: lane c forms corner c's term (in FP64, as
// window_height_regs), lane 0 adds them pairwise in corner order and forms the
// height and the log record.
template <int DIM>
__device__ __forceinline__ void chain_height(const Grp &g, GroupFixed<float> *fx, const Step &st, long long step,
                                             const DepositLog &log) {
  const GridDev &gd = fx->wd.g;
  double term = 0;
  if (g.lane < (1 << DIM) && fx->wd.method != ABP_METHOD_MABP) {  // mABP hills: fixed height
    double w = 1;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      const double f = (double)st.f[k];
      w *= ((g.lane >> k) & 1) ? f : 1.0 - f;
    }
    float4 ca, cb;
    rec_load<DIM>(node_ptr<DIM>(gd, corner_node<float, DIM>(gd, st, g.lane)), ca, cb);
    double v[4];
    rec_vals<float, DIM>(ca, cb, v);
    term = w * v[0];
  }
  double t[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) t[c] = c < (1 << DIM) ? __shfl_sync(0xffffffffu, term, c) : 0.0;
  if (g.lane == 0) window_height_out<float>(fx, st, t, step, log);
}

template <int DIM>
__device__ __forceinline__ void chain_body(const Grp &g, GroupFixed<float> *fx, Step *st, const SplitArgs &a) {
  const WalkerDev &wd = fx->wd;
  const int T = a.nsteps;
  const long long s0 = a.step0 + a.t0;
  const GroupLayout none{};
  // first deposit step of the block at or after t (a non-finite step deposits nothing)
  auto next_deposit = [&](int t) -> int {
    long long r = (s0 + t) % wd.stride;
    long long u = t + (r == 0 ? 0 : wd.stride - r);
    while (u < T && (st[u].flags & ABP_WFLAG_NONFINITE)) u += wd.stride;
    return u < T ? (int)u : T;
  };
  const int hw = g.nwarps - 1, tw = g.nwarps - 2;  // the warps of the height and of the tables
  int seg = 0;
  for (int dep = next_deposit(0);; dep = next_deposit(dep + 1)) {
    // on the grid as it is now, side by side: the look-ups of the steps since
    // the last deposit, the next deposit's height, its tables
    if (dep < T && g.warp == hw) {
      chain_height<DIM>(g, fx, st[dep], s0 + dep, a.log);
    } else if (dep < T && g.warp == tw) {
      window_dep_axis<float>(warp_grp(g), fx, st[dep]);
      __syncwarp();
      build_tables<float>(warp_grp(g), fx);
    } else {
      const int nl = dep < T ? tw * 32 : g.G;
      for (int q = seg + g.t; q < dep; q += nl) step_lookup<DIM>(wd, st + q);
    }
    if (dep == T) break;
    g.sync();
    deposit_stencil<float, false, 4>(g, fx, none, nullptr);
    g.sync();
    seg = dep;
  }
}

__device__ __forceinline__ void chain_any(const Grp &g, GroupFixed<float> *fx, Step *st, const SplitArgs &a) {
  if (fx->wd.g.d == 1)
    chain_body<1>(g, fx, st, a);
  else if (fx->wd.g.d == 2)
    chain_body<2>(g, fx, st, a);
  else
    chain_body<3>(g, fx, st, a);
}

// One CTA per walker. Bound by the chain of deposits: two rounds of grid
// reads (the height's corners, the stencil) and their barriers each.
__global__ void __launch_bounds__(kChainThreads, 1) k_sp_chain(SplitArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  const Grp g = cta_grp();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  load_words(g, &fx->wd, a.table[blockIdx.x].wd, (int)(sizeof(WalkerDev) / 4));
  g.sync();
  const WalkerDev &wd = fx->wd;
  if (wd.method == ABP_METHOD_MABP) return;  // k_sp_hist's
  if (a.terms && a.t0 == 0) 
    list_atom_terms(g, wd, atom_terms_of(a, blockIdx.x), atom_counts_of(a, blockIdx.x, wd.natoms));
  Step *st = walker_steps_of(a, blockIdx.x);
  chain_any(g, fx, st, a);
  g.sync();
  if (a.last && g.t == 0) state_out(wd, st[a.nsteps - 1], a.step0 + a.t0 + a.nsteps - 1);
}

// ---------------------------------------------------------------- a3 + a4, mABP

struct HistShared {
  float2 tab[kMaxCv][2 * kRMax + 2];  // per axis offset: the hill's factor (axis 0: times its height), -> derivative;
                                      // 0 past the stencil
  int4 walk[kHistWin];                // per step: its stencil's first node in the union's coordinates; w: todo
  int c[kMaxCv][kHistWin];            // per step: its node
  unsigned char todo[kHistWin];       // bit 0: deposits; bit 1: reads a node of the union; bit 2: reads outside it
  float raw[kHistWin][4];             // per step: the raw histograms at its node
};

// Slice blockIdx.y of a.slices of one mABP walker's grid (its nodes j of the
// last axis with j % slices == blockIdx.y): every hill of the block on them,
// in step order, and the look-ups that fall on them. Up to kHistWin steps at a
// time (fewer while their stencils' union exceeds kMabpUnion nodes): each
// thread keeps a node of the slice in registers, walks the hills, and stores
// the node once.
template <int DIM>
__device__ __forceinline__ void hist_body(const Grp &g, GroupFixed<float> *fx, HistShared *hs, Step *st,
                                          const SplitArgs &a) {
  constexpr int rb = DIM > 1 ? 32 : 16, U = 4;
  const WalkerDev &wd = fx->wd;
  const GridDev &gd = wd.g;
  const int slice = blockIdx.y, S = gridDim.y;
  const long long s0 = a.step0 + a.t0;
  int R[DIM], wrap[DIM], n[DIM];
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    R[k] = wd.R[k];
    n[k] = gd.n[k];
    wrap[k] = gd.periodic[k] ? gd.n[k] : 0;
  }
  if (g.t < DIM) {
    fx->da[g.t] = 0;
    fx->dc[g.t] = 0;
    fx->df[g.t] = 0;
  }
  g.sync();
  build_tables<float>(g, fx);  // node-centred: the same for every hill
  g.sync();
  const float h = (float)wd.w;
#pragma unroll
  for (int k = 0; k < DIM; ++k)
    for (int o = g.t; o < 2 * R[k] + 2; o += g.G)
      hs->tab[k][o] = o > 2 * R[k] ? make_float2(0.f, 0.f)
                                   : make_float2(k == 0 ? __fmul_rn(h, fx->tabG[k][o]) : fx->tabG[k][o], fx->tabD[k][o]);
  unsigned char *rec = reinterpret_cast<unsigned char *>(gd.rec);
  for (int t0 = 0; t0 < a.nsteps;) {
    int nt = min(kHistWin, a.nsteps - t0);
    g.sync();  // the steps before are done with the shared arrays
    for (int j = g.t; j < nt; j += g.G) {
      const Step &s = st[t0 + j];
      const bool ok = !(s.flags & ABP_WFLAG_NONFINITE);
#pragma unroll
      for (int k = 0; k < DIM; ++k) hs->c[k][j] = ok ? s.da[k] : 0;
      hs->todo[j] = ok ? ((s0 + t0 + j) % wd.stride == 0 ? 1 : 0) | 4 : 0;
    }
    g.sync();
    // the union of the deposits' stencil boxes, per axis relative to the
    // first deposit's node (every warp forms the same)
    int org[DIM], span[DIM], nodes;
    for (;; nt >>= 1) {
      int c0[DIM], first = nt;
      {
        const bool d0 = g.lane < nt && (hs->todo[g.lane] & 1), d1 = g.lane + 32 < nt && (hs->todo[g.lane + 32] & 1);
        const unsigned m0 = __ballot_sync(0xffffffffu, d0), m1 = __ballot_sync(0xffffffffu, d1);
        if (m0)
          first = __ffs(m0) - 1;
        else if (m1)
          first = __ffs(m1) + 31;
      }
      nodes = 0;
      if (first == nt) break;
      nodes = 1;
      bool big = false;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        c0[k] = hs->c[k][first];
        int lo = 0, hi = 0;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int j = g.lane + 32 * half;
          if (j < nt && (hs->todo[j] & 1)) {
            int dd = hs->c[k][j] - c0[k];
            if (wrap[k]) {
              dd %= n[k];
              if (dd < 0) dd += n[k];
              if (2 * dd > n[k]) dd -= n[k];
            }
            lo = min(lo, dd);
            hi = max(hi, dd);
          }
        }
        lo = __reduce_min_sync(0xffffffffu, lo) - R[k];
        hi = __reduce_max_sync(0xffffffffu, hi) + R[k];
        if (wrap[k]) {
          if (hi - lo + 1 >= n[k]) {
            org[k] = 0;
            span[k] = n[k];
          } else {
            org[k] = ((c0[k] + lo) % n[k] + n[k]) % n[k];
            span[k] = hi - lo + 1;
          }
        } else {
          org[k] = max(c0[k] + lo, 0);
          span[k] = min(c0[k] + hi, n[k] - 1) - org[k] + 1;
        }
        big = big || (long long)nodes * span[k] > kMabpUnion;
        nodes = big ? nodes : nodes * span[k];
      }
      if (nt == 1) {  // a single stencil box, whatever its size
        nodes = 1;
#pragma unroll
        for (int k = 0; k < DIM; ++k) nodes *= span[k];
        break;
      }
      if (!big) break;
    }
    g.sync();  // every warp has the union
    // per step: its place in the union, or outside (a step past the last, to
    // fill up the walk's rounds, touches nothing)
    const int ntu = (nt + U - 1) / U * U;
    for (int j = g.t; j < ntu; j += g.G) {
      int todo = j < nt ? hs->todo[j] : 0;
      int b[3] = {0, 0, 0};
      if (todo) {
        bool in = nodes > 0;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          const int c = hs->c[k][j];
          if (nodes > 0) {
            int r = c - org[k];
            r += r < 0 ? wrap[k] : 0;
            in = in && r >= 0 && r < span[k];
            b[k] = c - R[k] - org[k];
            if (wrap[k]) b[k] = ((b[k] % n[k]) + n[k]) % n[k];
          }
        }
        todo = (todo & 1) | (in ? 2 : 4);
        hs->todo[j] = (unsigned char)todo;
      }
      hs->walk[j] = make_int4(b[0], b[1], b[2], todo);
    }
    g.sync();
    // look-ups outside the union, by the slice that owns the node
    for (int j = g.t; j < nt; j += g.G)
      if ((hs->todo[j] & 4) && hs->c[DIM - 1][j] % S == slice) {
        long long node = 0, mul = 1;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          node += mul * hs->c[k][j];
          mul *= n[k];
        }
        float4 ra, rbv;
        rec_load<DIM>(rec + chk_node(gd, node) * rb, ra, rbv);
        float v[4] = {0.f, 0.f, 0.f, 0.f};
        rec_vals<float, DIM>(ra, rbv, v);
#pragma unroll
        for (int q = 0; q < 4; ++q) hs->raw[j][q] = v[q];
      }
    if (nodes > 0) {
      // this slice's planes of the last axis: j = org + r (one wrap at most)
      // with j % S == slice, in up to two runs
      const int L = DIM - 1, pre = min(span[L], n[L] - org[L]);  // before the wrap
      const int f0 = ((slice - org[L]) % S + S) % S, k0 = f0 < pre ? (pre - f0 + S - 1) / S : 0;
      const int k1 = span[L] - pre > slice ? (span[L] - pre - slice + S - 1) / S : 0;
      int plane = 1;
#pragma unroll
      for (int k = 0; k < DIM - 1; ++k) plane *= span[k];
      const int mine = plane * (k0 + k1);
      for (int i = g.t; i < mine; i += g.G) {
        int q[DIM], r0 = i;
        long long node = 0, mul = 1;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          if (k < DIM - 1) {
            q[k] = r0 % span[k];
            r0 /= span[k];
          } else {
            q[k] = r0 < k0 ? f0 + r0 * S : pre + slice + (r0 - k0) * S;
          }
          int j = org[k] + q[k];
          if (j >= n[k]) j -= n[k];
          node += mul * j;
          mul *= n[k];
        }
        unsigned char *ptr = rec + chk_node(gd, node) * rb;
        float4 ra, rbv;
        rec_load<DIM>(ptr, ra, rbv);
        // U steps a round: their places and factors first, all independent,
        // then the additions in step order (a chain of one add a hill)
        for (int j0 = 0; j0 < ntu; j0 += U) {
          float G[U], dd[U][3];
          bool in[U], centre[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int4 w = hs->walk[j0 + u];
            const int b[3] = {w.x, w.y, w.z};
            in[u] = (w.w & 1) != 0;
            centre[u] = (w.w & 2) != 0;
            G[u] = 1.f;
            dd[u][0] = dd[u][1] = dd[u][2] = 0.f;
#pragma unroll
            for (int k = 0; k < DIM; ++k) {
              int r = q[k] - b[k];
              r += r < 0 ? wrap[k] : 0;
              const int o = (int)min((unsigned)r, (unsigned)(2 * R[k] + 1));
              in[u] = in[u] & (o <= 2 * R[k]);
              centre[u] = centre[u] & (r == R[k]);
              const float2 tv = hs->tab[k][o];
              G[u] = k == 0 ? tv.x : __fmul_rn(G[u], tv.x);
              dd[u][k] = tv.y;
            }
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            // a hill that misses the node leaves the record as it was
            float4 na = ra, nb = rbv;
            rmw_regs<float>(DIM, na, nb, G[u], dd[u][0], dd[u][1], dd[u][2]);
            if (in[u]) {
              ra = na;
              rbv = nb;
            }
            if (centre[u]) {  // the step's look-up
              float v[4] = {0.f, 0.f, 0.f, 0.f};
              rec_vals<float, DIM>(ra, rbv, v);
#pragma unroll
              for (int e = 0; e < 4; ++e) hs->raw[j0 + u][e] = v[e];
            }
          }
        }
        float4 *p = reinterpret_cast<float4 *>(ptr);
        p[0] = ra;
        if (rb == 32) p[1] = rbv;
      }
    }
    if (slice == 0 && g.t == 0 && a.log.rec)
      for (int j = 0; j < nt; ++j)
        if (hs->todo[j] & 1) window_height<float, DIM>(fx, st[t0 + j], s0 + t0 + j, a.log);
    g.sync();
    for (int j = g.t; j < nt; j += g.G) {
      if (!hs->todo[j] || hs->c[DIM - 1][j] % S != slice) continue;
      Step &s = st[t0 + j];
      float V, dv[3] = {0.f, 0.f, 0.f}, acc[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[e] = hs->raw[j][e];
      mabp_bias<float>(wd, acc, V, dv);
      s.V = V;
#pragma unroll
      for (int k = 0; k < DIM; ++k)
        s.dv[k] = add_rn(((s.clamped >> k) & 1) ? 0.f : dv[k], wall_grad<float>(wd, k, s.s[k], s.sl[k]));
    }
    t0 += nt;
  }
  g.sync();
  if (a.last) {
    const Step &s = st[a.nsteps - 1];
    const bool bad = (s.flags & ABP_WFLAG_NONFINITE) != 0;
    const int owner = bad ? 0 : s.da[DIM - 1] % S;
    if (slice == owner && g.t == 0) state_out(wd, s, s0 + a.nsteps - 1);
  }
}

__global__ void __launch_bounds__(kHistThreads) k_sp_hist(SplitArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  const Grp g = cta_grp();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  HistShared *hs = reinterpret_cast<HistShared *>(smem + fixed_bytes_f());
  load_words(g, &fx->wd, a.table[blockIdx.x].wd, (int)(sizeof(WalkerDev) / 4));
  g.sync();
  const WalkerDev &wd = fx->wd;
  if (wd.method != ABP_METHOD_MABP) return;  // k_sp_chain's
  if (a.terms && a.t0 == 0 && blockIdx.y == 0) 
    list_atom_terms(g, wd, atom_terms_of(a, blockIdx.x), atom_counts_of(a, blockIdx.x, wd.natoms));
  Step *st = walker_steps_of(a, blockIdx.x);
  if (wd.g.d == 1)
    hist_body<1>(g, fx, hs, st, a);
  else if (wd.g.d == 2)
    hist_body<2>(g, fx, hs, st, a);
  else
    hist_body<3>(g, fx, hs, st, a);
}

// ---------------------------------------------------------------- a5

// The force records of one step of a walker, or null where there is nothing
// to write (the walker's own buffer keeps the call's last step).
__device__ __forceinline__ float4 *force_out(const SplitArgs &a, const WalkerDev &wd, int idx, int t) {
  if (a.forces) return reinterpret_cast<float4 *>(a.forces) + a.foff[idx] + (a.t0 + t) * a.fstride;
  return a.last && t == a.nsteps - 1 ? reinterpret_cast<float4 *>(wd.fbuf) : nullptr;
}

// A window's forces from its step records: the Jacobian factors scaled by
// dV/ds into shared memory (as finish_lookup scales them), then one atom per
// thread over every nl-th step, its terms (the walker's table) in registers.
// a.serial: every step writes the same records, so one CTA per walker takes
// the windows in turn, an atom always on the same thread.
struct ForceRec {
  float jac[kMaxCv * 12];
};
__global__ void __launch_bounds__(kForceThreads) k_sp_force(SplitArgs a) {
  __shared__ ForceRec fr[kWinMax];
  __shared__ int flag[kWinMax];
  const int tid = threadIdx.x;
  const TableEntry te = a.table[blockIdx.x];
  const WalkerDev &wd = *te.wd;
  const int natoms = wd.natoms, d = wd.g.d;
  const AtomTerm<float> *terms = reinterpret_cast<const AtomTerm<float> *>(wd.aterms);
  const int mode = a.forces ? a.mode : ABP_FORCES_OVERWRITE;
  const Step *st = walker_steps_of(a, blockIdx.x);
  const int wfirst = a.serial ? 0 : blockIdx.y, wend = a.serial ? (a.nsteps + kWinMax - 1) / kWinMax : wfirst + 1;
  for (int w = wfirst; w < wend; ++w) {
    const int t0 = w * kWinMax, nt = min(kWinMax, a.nsteps - t0);
    if (nt <= 0) return;
    __syncthreads();
    for (int i = tid; i < nt * kMaxCv * 12; i += kForceThreads) {
      const int j = i / (kMaxCv * 12), q = i - j * (kMaxCv * 12), k = q / 12;
      if (k < d) fr[j].jac[q] = __fmul_rn((&st[t0 + j].jac[0][0])[q], st[t0 + j].dv[k]);
    }
    for (int j = tid; j < nt; j += kForceThreads) flag[j] = st[t0 + j].flags;
    __syncthreads();
    const int nl = a.serial ? 1 : max(1, kForceThreads / natoms);
    for (int i = tid; i < natoms * nl; i += kForceThreads) {
      const int at = nl > 1 ? i % natoms : i, lane0 = nl > 1 ? i / natoms : 0;
      const int ne = wd.acnt[at];
      float tw[kAtomTerms];
      int toff[kAtomTerms];
#pragma unroll
      for (int q = 0; q < kAtomTerms; ++q) {
        const AtomTerm<float> v = q < ne ? terms[(size_t)at * kAtomTerms + q] : AtomTerm<float>{0.f, 0};
        tw[q] = v.w;
        toff[q] = v.off;
      }
      for (int j = lane0; j < nt; j += nl) {
        float4 *fo = force_out(a, wd, te.idx, t0 + j);
        if (!fo) continue;
        fo += at;
        if (flag[j] & ABP_WFLAG_NONFINITE) {
          if (mode == ABP_FORCES_OVERWRITE) *fo = make_float4(0.f, 0.f, 0.f, 0.f);
          continue;
        }
        float f0 = 0.f, f1 = 0.f, f2 = 0.f;
#pragma unroll
        for (int q = 0; q < kAtomTerms; ++q)
          if (q < ne) {
            const float *v = fr[j].jac + toff[q];
            f0 = fma_rn(tw[q], v[0], f0);
            f1 = fma_rn(tw[q], v[1], f1);
            f2 = fma_rn(tw[q], v[2], f2);
          }
        if (a.serial)
          store_force<float>(fo, make_float4(f0, f1, f2, 0.f), mode);
        else
          store_force_stream<float>(fo, make_float4(f0, f1, f2, 0.f), mode);
      }
    }
  }
}

// kCnfSteps steps of kCnfThreads atoms of one walker with gradient records, an
// atom a thread: each step's terms (list_atom_terms) in order, the steps'
// records loaded together. Bound by the gradient records read and the forces
// written (DRAM).
constexpr int kCnfSteps = 4, kCnfThreads = 256;

__global__ void __launch_bounds__(kCnfThreads) k_sp_cnf(SplitArgs a) {
  __shared__ ForceRec fr[kCnfSteps];  // Jacobian factors (COM distances: scaled by dV/ds)
  __shared__ float dvs[kCnfSteps][kMaxCv];
  __shared__ int flag[kCnfSteps];
  const int tid = threadIdx.x;
  const TableEntry te = a.table[blockIdx.x];
  const WalkerDev &wd = *te.wd;
  const int natoms = wd.natoms, d = wd.g.d, i = blockIdx.z * kCnfThreads + tid;
  if (blockIdx.z * kCnfThreads >= natoms) return;
  const int2 *terms = atom_terms_of(a, blockIdx.x);
  const int ne = i < natoms ? atom_counts_of(a, blockIdx.x, natoms)[i] : 0;
  const int mode = a.forces ? a.mode : ABP_FORCES_OVERWRITE;
  const Step *st = walker_steps_of(a, blockIdx.x);
  const int bfirst = a.serial ? 0 : blockIdx.y, bend = a.serial ? (a.nsteps + kCnfSteps - 1) / kCnfSteps : bfirst + 1;
  for (int b = bfirst; b < bend; ++b) {
    const int t0 = b * kCnfSteps, nt = min(kCnfSteps, a.nsteps - t0);
    if (b > bfirst) __syncthreads();
    for (int e = tid; e < nt * kMaxCv * 12; e += kCnfThreads) {
      const int j = e / (kMaxCv * 12), q = e - j * (kMaxCv * 12), k = q / 12;
      if (k < d) {
        const float v = (&st[t0 + j].jac[0][0])[q];
        fr[j].jac[q] = wd.cv[k].type == ABP_CV_COM_DIST ? __fmul_rn(v, st[t0 + j].dv[k]) : v;
      }
    }
    if (tid < nt * kMaxCv) dvs[tid / kMaxCv][tid % kMaxCv] = st[t0 + tid / kMaxCv].dv[tid % kMaxCv];
    if (tid < nt) flag[tid] = st[t0 + tid].flags;
    __syncthreads();
    if (i >= natoms) continue;
    const float4 *J = reinterpret_cast<const float4 *>(a.jac) + ((size_t)blockIdx.x * a.nsteps + t0) * a.jstride;
    float f[kCnfSteps][3];
#pragma unroll
    for (int j = 0; j < kCnfSteps; ++j) f[j][0] = f[j][1] = f[j][2] = 0.f;
    int2 next = terms[i];
    for (int q = 0; q < ne; ++q) {
      const int2 t = next;
      if (q + 1 < ne) next = terms[(q + 1) * natoms + i];
      const int kind = t.x & 3, k = t.x >> 2;
      if (kind == kCn) {
        float4 r[kCnfSteps];
#pragma unroll
        for (int j = 0; j < kCnfSteps; ++j)
          if (j < nt) r[j] = __ldcs(J + (size_t)j * a.jstride + t.y);  // read once
#pragma unroll
        for (int j = 0; j < kCnfSteps; ++j)
          if (j < nt) {
            const float v = -dvs[j][k];
            f[j][0] = fma_rn(v, r[j].x, f[j][0]);
            f[j][1] = fma_rn(v, r[j].y, f[j][1]);
            f[j][2] = fma_rn(v, r[j].z, f[j][2]);
          }
      } else {
        // COM distance: the weight on the scaled separation; dihedral: -dV/ds on the atom's gradient row
        const float w = __int_as_float(t.y);
        const int off = 12 * k + (kind == kDih ? 3 * t.y : 0);
#pragma unroll
        for (int j = 0; j < kCnfSteps; ++j)
          if (j < nt) {
            const float v = kind == kDih ? -dvs[j][k] : w;
            const float *u = fr[j].jac + off;
            f[j][0] = fma_rn(v, u[0], f[j][0]);
            f[j][1] = fma_rn(v, u[1], f[j][1]);
            f[j][2] = fma_rn(v, u[2], f[j][2]);
          }
      }
    }
    float4 *fo = force_out(a, wd, te.idx, t0);
#pragma unroll
    for (int j = 0; j < kCnfSteps; ++j)
      if (j < nt) {
        float4 *o = a.forces ? fo + j * a.fstride : force_out(a, wd, te.idx, t0 + j);
        if (!o) continue;
        if (!(flag[j] & ABP_WFLAG_NONFINITE)) {
          const float4 v = make_float4(f[j][0], f[j][1], f[j][2], 0.f);
          if (a.serial)
            store_force<float>(o + i, v, mode);
          else
            store_force_stream<float>(o + i, v, mode);
        } else if (mode == ABP_FORCES_OVERWRITE) {
          o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
  }
}

// ---------------------------------------------------------------- short calls
//
// The same parts in one launch, one CTA per walker, for calls of a few steps
// (a host engine's one step per call): records and Jacobians stay in shared
// memory. Bound by latency: the descriptor, the lists and coordinates, the
// CVs, the grid's corners, one after the other. Descriptors and lists are read
// before the earlier work of the stream is waited for. One step of one walker
// of two 16-atom groups and a dihedral: 16.2 us with a group of the windowed
// form, 8.2 us here; of 16 pocket walkers of 40 x 400 pairs 22.6 -> 14.6 us.

// Up to kWinMax steps of a walker of k_sp_cv's kind.
__global__ void __launch_bounds__(kShortThreads) k_sp_short(SplitArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  const Grp g = cta_grp();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  const TableEntry te = a.table[blockIdx.x];
  load_words(g, &fx->wd, te.wd, (int)(sizeof(WalkerDev) / 4));
  g.sync();
  const WalkerDev &wd = fx->wd;
  const int natoms = wd.natoms, d = wd.g.d, nt = a.nsteps;
  const CvLayout L = cv_layout(natoms, wd.cv, d, nt);
  Step *st = reinterpret_cast<Step *>(smem + L.recs);
  float4 *xs = reinterpret_cast<float4 *>(smem + L.xs);
  stage_lists(g, wd, smem + L.lists, fx->ia, fx->ib, fx->wa, fx->wb);
  // this thread's atom's a5 terms
  const AtomTerm<float> *terms = reinterpret_cast<const AtomTerm<float> *>(wd.aterms);
  const int ne0 = g.t < natoms ? wd.acnt[g.t] : 0;
  AtomTerm<float> mine[kAtomTerms];
#pragma unroll
  for (int q = 0; q < kAtomTerms; ++q)
    mine[q] = q < ne0 ? terms[(size_t)g.t * kAtomTerms + q] : AtomTerm<float>{0.f, 0};
  chain_wait();
  const float4 *cin = reinterpret_cast<const float4 *>(a.coords) + a.coff[te.idx];
  for (Iter2 it(g.t, g.G, natoms); it.j < nt; it.next())
    cp_async16(xs + it.j * L.xst + it.i, cin + (long long)it.j * a.cstride + it.i);
  cp_async_commit();
  window_records(g, fx, xs, L.xst, st, nt, a.step0, a.ctr);
  chain_any(g, fx, st, a);
  g.sync();
  if (g.t == 0) state_out(wd, st[nt - 1], a.step0 + nt - 1);
  for (int i = g.t; i < nt * kMaxCv * 12; i += g.G) {
    const int j = i / (kMaxCv * 12), q = i - j * (kMaxCv * 12), k = q / 12;
    float *v = &st[j].jac[0][0] + q;
    if (k < d) *v = __fmul_rn(*v, st[j].dv[k]);
  }
  g.sync();
  const int mode = a.forces ? a.mode : ABP_FORCES_OVERWRITE;
  for (int at = g.t; at < natoms; at += g.G) {
    int ne = ne0;
    if (at != g.t) {
      ne = wd.acnt[at];
#pragma unroll
      for (int q = 0; q < kAtomTerms; ++q)
        mine[q] = q < ne ? terms[(size_t)at * kAtomTerms + q] : AtomTerm<float>{0.f, 0};
    }
    for (int j = 0; j < nt; ++j) {
      float4 *fo = force_out(a, wd, te.idx, j);
      if (!fo) continue;
      if (st[j].flags & ABP_WFLAG_NONFINITE) {
        if (mode == ABP_FORCES_OVERWRITE) fo[at] = make_float4(0.f, 0.f, 0.f, 0.f);
        continue;
      }
      float f0 = 0.f, f1 = 0.f, f2 = 0.f;
#pragma unroll
      for (int q = 0; q < kAtomTerms; ++q)
        if (q < ne) {
          const float *v = &st[j].jac[0][0] + mine[q].off;
          f0 = fma_rn(mine[q].w, v[0], f0);
          f1 = fma_rn(mine[q].w, v[1], f1);
          f2 = fma_rn(mine[q].w, v[2], f2);
        }
      store_force<float>(fo + at, make_float4(f0, f1, f2, 0.f), mode);
    }
  }
}

// Shared memory of k_sp_one: GroupFixed | step record | lists | A gradients |
// coordinates | gradient records | forces.
struct OneLayout {
  int rec, lists, lig, xs, jac, fs, total;
};
__host__ __device__ inline OneLayout one_layout(int natoms, const CvDev *cv, int d) {
  OneLayout L;
  L.rec = fixed_bytes_f();
  L.lists = up32(L.rec + (int)sizeof(Step));
  L.lig = L.lists + list_bytes(cv, d);
  L.xs = up32(L.lig + kCnWarps * cn_lig_floats(cv, d) * 4);
  L.jac = L.xs + natoms * 16;
  L.fs = L.jac + cn_records(cv, d) * 16;
  L.total = L.fs + natoms * 16;
  return L;
}

// One step of a walker of k_sp_cn's kind: the coordination numbers on the
// first four warps, COM distances on the fifth, dihedrals on the sixth.
__global__ void __launch_bounds__(kOneThreads) k_sp_one(SplitArgs a) {
  extern __shared__ __align__(32) unsigned char smem[];
  __shared__ float red[kCnWarps][2];
  const Grp g = cta_grp();
  GroupFixed<float> *fx = reinterpret_cast<GroupFixed<float> *>(smem);
  const TableEntry te = a.table[blockIdx.x];
  load_words(g, &fx->wd, te.wd, (int)(sizeof(WalkerDev) / 4));
  g.sync();
  const WalkerDev &wd = fx->wd;
  const int natoms = wd.natoms, d = wd.g.d;
  const OneLayout L = one_layout(natoms, wd.cv, d);
  Step *st = reinterpret_cast<Step *>(smem + L.rec);
  float *ligs = reinterpret_cast<float *>(smem + L.lig);
  float4 *x = reinterpret_cast<float4 *>(smem + L.xs), *J = reinterpret_cast<float4 *>(smem + L.jac);
  float4 *fs = reinterpret_cast<float4 *>(smem + L.fs);
  stage_lists(g, wd, smem + L.lists, fx->ia, fx->ib, fx->wa, fx->wb);
  for (int i = g.t; i < natoms; i += g.G) fs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  chain_wait();
  const float4 *cin = reinterpret_cast<const float4 *>(a.coords) + a.coff[te.idx];
  for (int i = g.t; i < natoms; i += g.G) cp_async16(x + i, cin + i);
  cp_async_commit();
  cp_async_wait_all();
  __syncthreads();
  float4 *fo = force_out(a, wd, te.idx, 0);
  const int mode = a.forces ? a.mode : ABP_FORCES_OVERWRITE;
  if (__syncthreads_or(!step_finite(x, natoms, g.t, g.G))) {
    if (mode == ABP_FORCES_OVERWRITE)
      for (int i = g.t; i < natoms; i += g.G) fo[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (g.t == 0) {
      wd.state->flags = ABP_WFLAG_NONFINITE;
      atomicAdd(&a.ctr->nonfinite, 1);
    }
    return;
  }
  const bool dep = a.step0 % wd.stride == 0;
  float4 *Jk = J;
  for (int k = 0; k < d; ++k) {
    const CvDev &c = wd.cv[k];
    if (c.type == ABP_CV_COM_DIST) {
      if (g.warp == kCnWarps) {
        float s = 0.f, sl = 0.f;
        const int fl = com_one_warp(c, fx->ia[k], fx->ib[k], fx->wa[k], fx->wb[k], x, g.lane, s, sl, st->jac[k]);
        if (g.lane == 0) window_cv_rec<float>(wd, k, s, sl, fl, dep, *st);
      }
    } else if (c.type == ABP_CV_DIHEDRAL) {
      if (g.t == g.G - 1) window_cv<float>(fx, x, k, dep, *st);
    } else {
      const float c6 = -6.f * (float)c.inv_r0sq;
      if (g.warp < kCnWarps) {
        float h[1], l[1];
        cn_warp_any(c, fx->ia[k], fx->ib[k], x, Jk + c.na, ligs + g.warp * c.na * 3, false, g.lane, 8 * g.warp,
                    8 * kCnWarps, h[0], l[0]);
        warp_sum_ff<1>(h, l);
        if (g.lane == 0) {
          red[g.warp][0] = h[0];
          red[g.warp][1] = l[0];
        }
      }
      __syncthreads();
      if (g.t == 0) {
        float sh = red[0][0], sl = red[0][1];
#pragma unroll
        for (int v = 1; v < kCnWarps; ++v) ff_add<float>(sh, sl, red[v][0], red[v][1]);
        window_cv_rec<float>(wd, k, sh, sl, 0, dep, *st);
      }
      for (int i = g.t; i < c.na; i += g.G) {
        float s3[3];
#pragma unroll
        for (int e = 0; e < 3; ++e) {
          s3[e] = ligs[3 * i + e];
#pragma unroll
          for (int v = 1; v < kCnWarps; ++v) s3[e] = __fadd_rn(s3[e], ligs[(v * c.na + i) * 3 + e]);
        }
        Jk[i] = make_float4(__fmul_rn(c6, s3[0]), __fmul_rn(c6, s3[1]), __fmul_rn(c6, s3[2]), 0.f);
      }
      __syncthreads();  // the scratch is free again
      Jk += c.na + c.nb;
    }
  }
  __syncthreads();
  if (g.t == 0) step_flags<float>(d, dep, *st);
  __syncthreads();
  chain_any(g, fx, st, a);
  g.sync();
  if (g.t == 0) state_out(wd, *st, a.step0);
  // a5: list by list (an atom appears at most once in a list), CV by CV
  int jpos = 0;
  for (int k = 0; k < d; ++k) {
    const CvDev &c = wd.cv[k];
    const bool com = c.type == ABP_CV_COM_DIST, cn = c.type == ABP_CV_COORD;
    const float dv = st->dv[k];
    const float u0 = __fmul_rn(st->jac[k][0], dv), u1 = __fmul_rn(st->jac[k][1], dv), u2 = __fmul_rn(st->jac[k][2], dv);
    for (int lst = 0; lst < (com || cn ? 2 : 1); ++lst) {
      const int n = lst ? c.nb : (com || cn ? c.na : 4);
      const int32_t *list = lst ? fx->ib[k] : fx->ia[k];
      for (int i = g.t; i < n; i += g.G) {
        float w, v0, v1, v2;
        if (com) {
          w = lst ? -fx->wb[k][i] : fx->wa[k][i];
          v0 = u0;
          v1 = u1;
          v2 = u2;
        } else if (cn) {
          const float4 j = J[jpos + (lst ? c.na : 0) + i];
          w = -dv;
          v0 = j.x;
          v1 = j.y;
          v2 = j.z;
        } else {
          w = -dv;
          v0 = st->jac[k][3 * i];
          v1 = st->jac[k][3 * i + 1];
          v2 = st->jac[k][3 * i + 2];
        }
        float4 &f = fs[list[i]];
        f.x = fma_rn(w, v0, f.x);
        f.y = fma_rn(w, v1, f.y);
        f.z = fma_rn(w, v2, f.z);
      }
      __syncthreads();
    }
    if (cn) jpos += c.na + c.nb;
  }
  for (int i = g.t; i < natoms; i += g.G) store_force<float>(fo + i, fs[i], mode);
}

}  // namespace

// ---------------------------------------------------------------- host side

size_t split_step_bytes() { return sizeof(Step); }

// 8-byte words of a walker's atom terms and counts (an atom's list entries fit
// kAtomTerms slots: at most two lists per CV).
int split_term_words(const WalkerDev &hd) { return hd.natoms * kAtomTerms + (hd.natoms + 1) / 2; }

int split_jac_records(const WalkerDev &hd) { return cn_records(hd.cv, hd.g.d); }

bool split_eligible(const WalkerDev &hd, bool win) {
  const int limit = 227 * 1024;
  if (win) return hd.aterms != nullptr;
  return cn_bytes(hd.cv, hd.g.d, hd.natoms) <= limit;
}

void split_shape(const WalkerDev &hd, bool win, SplitShape *s) {
  if (win) {
    const int W = window_steps(hd.natoms, hd.cv, hd.g.d, 16);
    s->cv_smem = max(s->cv_smem, cv_layout(hd.natoms, hd.cv, hd.g.d, W).total);
    s->win = s->win == 0 ? W : min(s->win, W);
  } else {
    s->cv_smem = max(s->cv_smem, cn_bytes(hd.cv, hd.g.d, hd.natoms));
    s->staged = s->staged && hd.natoms * 16 <= kCnStage;
    for (int k = 0; k < hd.g.d; ++k) s->long_cn = s->long_cn || (hd.cv[k].type == ABP_CV_COORD && hd.cv[k].na > 40);
  }
  if (hd.method == ABP_METHOD_MABP)
    s->mabp += 1;
  else
    s->wt += 1;
  s->min_dim = s->min_dim == 0 ? hd.g.d : min(s->min_dim, hd.g.d);
  s->max_atoms = max(s->max_atoms, hd.natoms);
}

int short_smem(const WalkerDev &hd, bool win, int nsteps) {
  return win ? cv_layout(hd.natoms, hd.cv, hd.g.d, nsteps).total : one_layout(hd.natoms, hd.cv, hd.g.d).total;
}

cudaError_t launch_short(const SplitArgs &a, bool win, int smem, LaunchTimer *tm, cudaStream_t st) {
  void (*k)(SplitArgs) = win ? k_sp_short : k_sp_one;
  const char *name = win ? "k_sp_short" : "k_sp_one";
  cudaError_t e = smem_attr(reinterpret_cast<const void *>(k), smem);
  if (e != cudaSuccess) return e;
  NvtxRange nv(name);
  if (tm) tm->begin(name, st);
  e = launch_chained(k, a.nw, win ? kShortThreads : kOneThreads, smem, st, a);
  if (tm) tm->end(name, st);
  return e;
}

cudaError_t launch_split(const SplitArgs &a0, const SplitShape &s, int sms, LaunchTimer *tm, cudaStream_t st) {
  SplitArgs a = a0;
  cudaError_t e = cudaSuccess;
  auto run = [&](const char *name, void (*k)(SplitArgs), dim3 grid, int threads, size_t smem) {
    if (e != cudaSuccess) return;
    if ((e = smem_attr(reinterpret_cast<const void *>(k), smem)) != cudaSuccess) return;
    NvtxRange nv(name);
    if (tm) tm->begin(name, st);
    k<<<grid, threads, smem, st>>>(a);
    if (tm) tm->end(name, st);
    e = cudaGetLastError();
  };
  const unsigned nw = (unsigned)a.nw;
  const bool win = s.win > 0;
  if (win) {
    run("k_sp_cv", k_sp_cv, dim3(nw, (a.nsteps + s.win - 1) / s.win), kCvThreads, s.cv_smem);
  } else {
    // one step a warp once the batch has a step for every warp the chip
    // holds (16 an SM), in runs of up to kCnBatch consecutive steps while three
    // rounds of warps remain; below that one step a CTA
    const long long items = (long long)a.nw * a.nsteps, slots = 16ll * sms;
    a.chunk = (int)max(1ll, min((long long)kCnBatch, items / max(1ll, 3 * slots)));
    const bool per_warp = items >= slots;
    void (*const ks[2][2][2])(SplitArgs) = {  // [per_warp][staged][long_cn]
        {{k_sp_cn<false, false, false>, k_sp_cn<false, false, true>},
         {k_sp_cn<false, true, false>, k_sp_cn<false, true, true>}},
        {{k_sp_cn<true, false, false>, k_sp_cn<true, false, true>},
         {k_sp_cn<true, true, false>, k_sp_cn<true, true, true>}}};
    void (*k)(SplitArgs) = ks[per_warp][s.staged][s.long_cn];
    run("k_sp_cn", k, dim3(nw, per_warp ? (a.nsteps + a.chunk * kCnWarps - 1) / (a.chunk * kCnWarps) : a.nsteps),
        kCnThreads, s.cv_smem);
  }
  // a wide CTA takes a stencil in one round; with several walkers an SM, half of it
  if (s.wt) run("k_sp_chain", k_sp_chain, dim3(nw), a.nw <= sms ? kChainThreads : kChainThreads / 2, fixed_bytes_f());
  if (s.mabp) {
    // slices of the last axis (a 1D stencil is too small to cut): about four CTAs an SM
    const int S = s.min_dim < 2 ? 1 : max(1, min(8, 4 * sms / max(1, a.nw)));
    run("k_sp_hist", k_sp_hist, dim3(nw, S), kHistThreads, fixed_bytes_f() + sizeof(HistShared));
  }
  if (win) {
    run("k_sp_force", k_sp_force, dim3(nw, a.serial ? 1 : (a.nsteps + kWinMax - 1) / kWinMax), kForceThreads, 0);
  } else {
    run("k_sp_cnf", k_sp_cnf,
        dim3(nw, a.serial ? 1 : (a.nsteps + kCnfSteps - 1) / kCnfSteps, (s.max_atoms + kCnfThreads - 1) / kCnfThreads),
        kCnfThreads, 0);
  }
  return e;
}

}  // namespace abp
