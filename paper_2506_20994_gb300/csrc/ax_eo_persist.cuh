// Persistent fp64-accurate element operator (Listing 2) for the operator
// handle: the even-odd double-float schedule of ax_df64_eo.cuh, one element
// per CTA at a time, with the element's geometry streamed into shared memory
// by the bulk-copy engine one element ahead.
//
// Why a second schedule: the even-odd kernel that reads its geometry with
// per-thread loads spends its time waiting on those loads (16 warps per SM
// at 128 registers, two geometry stages held in registers) and reaches only
// half of the HBM bandwidth although its arithmetic would allow more.  Here
//  * each CTA loops over elements e = blockIdx.x, + gridDim.x, ...; while it
//    computes element e, one `cp.async.bulk` (completion on an mbarrier)
//    brings the next element's prepared geometry (56 lx^3 bytes, contiguous)
//    into shared memory, and every thread's u values of the next element are
//    already loaded into registers, so no phase waits on global memory;
//  * the element's (lx/2)^3 mirror octants get two threads each (thread
//    2t + c owns the four points {i', N-i'} x {j', N-j'} x {k} with k = k'
//    for c = 0 and N - k' for c = 1); pairs along i and j stay inside a
//    thread, pairs along k are formed with one shuffle with the partner lane;
//  * the line buffers of the three directions are XOR-swizzled at lx = 8
//    (four 16-byte entries per line, no padding, conflict-free reads and
//    writes); four CTAs of 124 registers per SM (measured faster than five
//    of 96: the double-float chains want the registers more than the warps).
// The arithmetic is that of the even-odd kernel on prepared geometry
// (double-float pairs, packed f32x2, the two half-size sums of each 1-D
// contraction as the two lanes).  Elements outside the double-float range
// (guard.cuh) are recomputed with fp64 units from the caller's fp64 arrays;
// matrices that are not centro-antisymmetric never reach the handle's kernel
// (the handle checks them when it is created).  The same body also runs on
// the caller's raw fp64 arrays (RAW, ax_helm): seven bulk copies per
// element, geometry split per apply, matrices and exponent window checked in
// the kernel.  Lines at lx = 6 and 10 rotate their entries (lpos).
#pragma once

#include "common.cuh"
#include "dispatch.h"
#include "df64.cuh"
#include "guard.cuh"

namespace ax {
namespace eop {

template <int LX>
struct Cfg {
  static constexpr int H = LX / 2, N = LX - 1, H2 = H * H, H3 = H2 * H;
  static constexpr int NT = 2 * H3;                // threads per element
  static constexpr int NTB = (NT + 31) / 32 * 32;  // block size
  static constexpr int NW = NTB / 32;
  static constexpr int N3 = LX * LX * LX;
  static constexpr bool SWZ = H == 4;              // swizzled, unpadded lines
  // 16-byte entry slots per line (see lpos)
  static constexpr int LS = SWZ ? 4 : H + 1;
  static constexpr int DE = LX * LX * LS;          // entries per direction
  static constexpr int GE = 2 * 7 * NT;            // geometry entries per element
  static constexpr unsigned GBYTES = GE * 16u;     // = 56 lx^3
  static constexpr int CS = H + 1;                 // padded coefficient row (dd2 entries)
  static constexpr size_t COEF_BYTES = 2 * H * CS * 16 + 2 * H2 * 8;
  static constexpr size_t OFF_LINES = (COEF_BYTES + 127) / 128 * 128;
  static constexpr size_t LINE_BYTES = 3 * (size_t)DE * 16;
  static constexpr size_t OFF_G = OFF_LINES + (LINE_BYTES + 127) / 128 * 128;
  static constexpr size_t OFF_MISC = OFF_G + GBYTES;
  // mbarrier (8 B, padded to 16), one key slot and one dot slot per warp
  // (raw-array form: the key slots of G and h1 share the dot slots, and 16
  // bytes hold the matrices' largest entry and symmetry defect)
  static constexpr size_t SMEM = OFF_MISC + 16 + NW * 8 + NW * 8 + 16;
  // resident CTAs per SM the launch bounds ask for
  static constexpr int MINB = LX == 6 ? 8 : LX == 8 ? 4 : LX == 10 ? 2 : 1;
  // the fused direction update may carry the solver's x update (EopUpd::x)
  static constexpr bool XUP = eop_x_update(LX);
  static_assert(LINE_BYTES >= 3 * (size_t)N3 * 8, "fallback scratch must fit the lines");
};

// Entry `ent` of line L.  At lx = 8 (L = 8 * outer + inner) the line slot
// swaps neighbours when bit 3 of L is set and the entry is XOR-ed with bits 1
// and 3 of L: every line read and write of the kernel then touches each
// 16-byte bank group at most once per wavefront's worth of distinct entries.
// At lx = 6 and lx = 10 (lines padded to 4 and 6 slots) the entries rotate
// within the line by an offset that depends on the line (lx = 6: L + L / 6;
// lx = 10: 5 (L / 10)): a model of the kernel's warp accesses (half-warp
// phases of 16-byte accesses) gives 198 wavefronts per element pass against
// 556 unrotated at lx = 6, and 1226 against 1848 at lx = 10.
// ROT10: the lx = 10 rotation (the single-mesh kernel; in the batched
// kernel's 128-register slots it measured slower, 1.74 against 1.66 ms on the
// benchmark batch, and is left out there).
template <int LX, bool ROT10 = true>
AX_D int lpos(int L, int ent) {
  if constexpr (Cfg<LX>::SWZ) {
    const int b3 = (L >> 3) & 1;
    return (L ^ b3) * 4 + (ent ^ (((L >> 1) & 1) | (b3 << 1)));
  } else if constexpr (LX == 6) {
    return L * 4 + ((ent + L + L / 6) & 3);
  } else if constexpr (LX == 10 && ROT10) {
    return L * 6 + (ent + (L / 10) * 5) % 6;
  } else {
    return L * Cfg<LX>::LS + ent;
  }
}

AX_D uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
AX_D void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// One bulk copy global -> shared of `bytes` (16-byte aligned, multiple of
// 16), completing on the mbarrier's current phase (single arrival + bytes).
AX_D void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
// The same as several copies on one phase: one arrival announcing all
// bytes, then the copies (bulk_copy).
AX_D void mbar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
AX_D void bulk_copy(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}
// Generic-proxy reads of a buffer before the bulk engine rewrites it.
AX_D void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
AX_D unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// A wait gives up after kWaitNs of global time (or `limit` polls, a
// backstop; each poll may suspend the thread for a short, bounded time).
constexpr unsigned long long kWaitNs = 2000000000ull;  // 2 s
constexpr int kWaitLimit = 1 << 30;
// Waits for the mbarrier phase with the given parity; false when it gave up.
AX_D bool mbar_wait(uint32_t bar, uint32_t parity, int limit) {
  unsigned long long t0 = 0ull;
  for (int it = 0; it < limit; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if ((it & 1023) == 1023) {  // the clock only once a wait is long
      const unsigned long long t = global_ns();
      if (t0 == 0ull)
        t0 = t;
      else if (t - t0 > kWaitNs)
        return false;
    }
  }
  return false;
}

// exchange of one pair with the partner lane (tid ^ 1)
AX_D df::df2 xchg(df::df2 v) {
  return df::df2{__shfl_xor_sync(0xffffffffu, v.hi, 1), __shfl_xor_sync(0xffffffffu, v.lo, 1)};
}

// Operands of one mesh for the persistent body: w = Ax(u), the prepared
// geometry (gp) and its per-element u exponent ranges, the staged
// coefficient block, and the fp64 arrays an element falls back to.
struct EopMesh {
  double *w = nullptr;
  const double *u = nullptr;
  const df::dd2 *coef = nullptr, *gp = nullptr;
  const uint2 *urange = nullptr;
  guard::RawGeo raw{};
  const double *dx = nullptr, *dxt = nullptr;
  // HB: h2 .* B of the Helmholtz form, w = Ax(u) + hb .* u
  const double *hb = nullptr;
  // testing aid (ax_op_inject_copy_loss): this element's geometry copy is
  // never issued, so its wait runs out; -1: none
  long long drop = -1;
};

// Solver operands of the fused direction update (PUPD): pw = minv .* r
// (+ corr when use_corr) + beta pw, formed in place in front of the apply;
// x (may be null) += alpha pw with the old pw: the previous step's solution
// update, whose read of pw is this one's (at 56 % of HBM the apply has the
// bandwidth to spare that the solver's vector kernels lack); only at the orders
// of eop_x_update.  The vectors are read through L1: at lx 6 and 10 an
// element's rows are no whole 32-byte sectors, and past L1 each sector came
// twice (an apply at 26^3 elements, lx 10: 595 -> 554 us; an iteration at 32^3,
// lx 8: 632 -> 619 us).  In a chained launch this is safe because only the
// solver loops launch this form, behind a kernel that reads these vectors past
// L1 (the update or the dots), and that kernel's own launch has emptied L1 of
// what the apply before it had read.
struct EopUpd {
  double *pw;
  const double *r, *minv, *corr;
  double *x;
  double alpha, beta;
  bool use_corr;
};

// A position in a body's element sequence: item index and element offset.
struct EopPos {
  int it;
  long long off;
};

// The operator handle's sequence: elements blockIdx.x, + gridDim.x, ... of
// one mesh.  The mesh operands are held by value (copies of kernel
// parameters), so the compiler reads them from the constant bank; through a
// pointer every per-element access would be a load.
struct SeqOne {
  static constexpr bool kRotate10 = true;  // line layout, see lpos
  static constexpr bool kOneMesh = true;   // coefficients staged once
  EopMesh m;
  long long nelv;
  AX_D bool first(EopPos &p) const {
    p = EopPos{0, (long long)blockIdx.x};
    return p.off < nelv;
  }
  AX_D bool advance(const EopPos &p, EopPos &q) const {
    q = EopPos{0, p.off + (long long)gridDim.x};
    return q.off < nelv;
  }
  AX_D int mesh_of(const EopPos &) const { return 0; }
  AX_D long long elem(const EopPos &p) const { return p.off; }
  AX_D const EopMesh &mesh(int) const { return m; }
};

// Persistent even-odd body over the element sequence `seq` of one group of
// NTB threads (`tid` in [0, NTB)) with `sm` its shared memory (Cfg<LX>::SMEM
// bytes, 128-byte aligned).  sync() / sync_and(p) synchronise exactly that
// group (the second also ANDs a predicate over it).  DOT: adds this thread's
// share of u . w to dsum.  PUPD: u is not an input; phase 1 forms the
// solver's next direction in place (EopUpd), fp64 with explicit roundings,
// and the operator is applied to it.  err: set to 1 if a staged copy never
// arrived (the body then stops).
// RAW: the geometry comes straight from the caller's fp64 arrays (M.raw;
// seven bulk copies per element, split per apply), the coefficients and the
// matrices' exponent field and symmetry are formed here from M.dx, M.dxt,
// and each element's exponent window is checked from its own values; M.gp,
// M.coef and M.urange are not used.  (ax_helm on fp64 arrays.)
// HB: the Helmholtz mass term, w += M.hb .* u with fp64 units as w is stored.
// As a pass of its own it moved 32 bytes a point more (4096 elements, lx = 10:
// 134.9 us a call, 118.5 so; 109 with the shorter split).
// ready(): called once, after the set-up that needs no other kernel's results
// (the first element's prepared geometry and the coefficients, both the
// handle's own) and before everything else; RAW calls it first.
template <int LX, bool DOT, bool PUPD, bool RAW = false, bool DROP = false, bool HB = false,
          class Seq, class Sync, class SyncAnd, class Ready>
AX_D void eop_run(unsigned char *sm, int tid, const Seq &seq, Sync sync, SyncAnd sync_and,
                  int *err, EopUpd &up, double &dsum, Ready ready) {
  static_assert(!RAW || (!DOT && !PUPD), "the raw-array form is the plain apply");
  static_assert(!HB || (!DOT && !PUPD && !RAW), "the mass term joins the handle's plain apply");
  using namespace df;
  using C = Cfg<LX>;
  constexpr int H = C::H, N = C::N, H2 = C::H2, NT = C::NT, NW = C::NW, N3 = C::N3;
  constexpr int CS = C::CS;
  dd2 *cf = reinterpret_cast<dd2 *>(sm);  // [H][CS] (P, M) of D, rows padded
  dd2 *tf = cf + H * CS;                  // [H][CS] (P, M) of D^T
  u64 *cn = reinterpret_cast<u64 *>(tf + H * CS);  // [H][H] negated heads
  u64 *tn = cn + H2;
  // line buffer: per direction [k][j] (r), [k][i] (s), [j][i] (t)
  dd2 *Lb = reinterpret_cast<dd2 *>(sm + C::OFF_LINES);
  dd2 *Gs = reinterpret_cast<dd2 *>(sm + C::OFF_G);
  const uint32_t bar = smem_u32(sm + C::OFF_MISC);
  unsigned *kslot = reinterpret_cast<unsigned *>(sm + C::OFF_MISC + 16);
  unsigned *gslot = reinterpret_cast<unsigned *>(sm + C::OFF_MISC + 16 + NW * 8);  // RAW
  unsigned long long *drec =
      reinterpret_cast<unsigned long long *>(sm + C::OFF_MISC + 16 + NW * 16);  // RAW
  bool raw_ok = true;  // RAW: matrices centro-antisymmetric, finite
  int raw_fd = 0;      // RAW: their exponent field

  const bool real = tid < NT;
  const int t = real ? tid >> 1 : 0, c = tid & 1;
  const int ip = t % H, jp = (t / H) % H, kp = t / H2;
  const int kk = c ? N - kp : kp;
  auto pidx = [&](int b, int a) __attribute__((always_inline)) {
    return (kk * LX + (b ? N - jp : jp)) * LX + (a ? N - ip : ip);
  };
  auto lineR = [&](int b) __attribute__((always_inline)) { return kk * LX + (b ? N - jp : jp); };
  auto lineS = [&](int a) __attribute__((always_inline)) { return kk * LX + (a ? N - ip : ip); };
  auto lineT = [&](int b, int a) __attribute__((always_inline)) { return (b ? N - jp : jp) * LX + (a ? N - ip : ip); };
  auto eo_pair = [](df2 v0, df2 v1) __attribute__((always_inline)) {
    return dsum2(dd2{pk(v0.hi, v0.hi), pk(v0.lo, v0.lo)},
                 dd2{pk_pm(v1.hi), pk_pm(v1.lo)});
  };
  // half-size contractions of line L of `lines`: (y at row, y at N-row)
  auto contract = [&](const dd2 *lines, int L, const dd2 *cof, const u64 *nco, int row,
                      df2 &y_lo, df2 &y_hi) __attribute__((always_inline)) {
    acc2 a = prod2(cof[row * CS], nco[row * H], lines[lpos<LX, Seq::kRotate10>(L, 0)]);
#pragma unroll
    for (int l = 1; l < H; ++l)
      mac2(a, cof[row * CS + l], nco[row * H + l], lines[lpos<LX, Seq::kRotate10>(L, l)]);
    const float Es = lx_(a.s), Ec = lx_(a.c), Os = ly_(a.s), Oc = ly_(a.c);
    const dd2 r = dsum2(dd2{pk(Os, Os), pk(Oc, Oc)}, dd2{pk_pm(Es), pk_pm(Ec)});
    y_lo = df2{lx_(r.hi), lx_(r.lo)};
    y_hi = df2{ly_(r.hi), ly_(r.lo)};
  };
  // the three directions' lines of one field (v[b][a] at this thread's points)
  auto publish = [&](dd2 *Ar, df2 (&vr)[2][2], df2 (&vs)[2][2], df2 (&vt)[2][2])
                     __attribute__((always_inline)) {
    dd2 *As = Ar + C::DE, *At = As + C::DE;
    // k-pairs: this thread forms the entries of lines (b = c, a); it needs the
    // partner's values there, the partner its values at b = 1 - c
    // (selects, not vt[1 - c]: a run-time index would put the array in local memory)
    df2 o0 = xchg(c ? vt[0][0] : vt[1][0]), o1 = xchg(c ? vt[0][1] : vt[1][1]);
    if (real) {
#pragma unroll
      for (int b = 0; b < 2; ++b) Ar[lpos<LX, Seq::kRotate10>(lineR(b), ip)] = eo_pair(vr[b][0], vr[b][1]);
#pragma unroll
      for (int a = 0; a < 2; ++a) As[lpos<LX, Seq::kRotate10>(lineS(a), jp)] = eo_pair(vs[0][a], vs[1][a]);
      At[lpos<LX, Seq::kRotate10>(lineT(c, 0), kp)] = c ? eo_pair(o0, vt[1][0]) : eo_pair(vt[0][0], o0);
      At[lpos<LX, Seq::kRotate10>(lineT(c, 1), kp)] = c ? eo_pair(o1, vt[1][1]) : eo_pair(vt[0][1], o1);
    }
  };
  // contractions of the three directions into this thread's points
  auto contract_all = [&](const dd2 *Ar, const dd2 *cof, const u64 *nco, df2 (&yr)[2][2],
                          df2 (&ys)[2][2], df2 (&yt)[2][2]) __attribute__((always_inline)) {
    const dd2 *As = Ar + C::DE, *At = As + C::DE;
#pragma unroll
    for (int b = 0; b < 2; ++b) contract(Ar, lineR(b), cof, nco, ip, yr[b][0], yr[b][1]);
#pragma unroll
    for (int a = 0; a < 2; ++a) contract(As, lineS(a), cof, nco, jp, ys[0][a], ys[1][a]);
#pragma unroll
    for (int a = 0; a < 2; ++a) {
      df2 y0, y1;  // at k = k' and k = N - k' of point (b = c, a)
      contract(At, lineT(c, a), cof, nco, kp, y0, y1);
      const df2 own = c ? y1 : y0;
      const df2 recv = xchg(c ? y0 : y1);  // the partner's line, at this thread's k
      yt[0][a] = c ? recv : own;
      yt[1][a] = c ? own : recv;
    }
  };

  auto load_coef = [&](const EopMesh &M) __attribute__((always_inline)) {
    if constexpr (RAW) {
      // what the handle's set-up does on the host (eop_coefficients)
      if (tid == 0) {
        drec[0] = 0ull;
        drec[1] = 0ull;
      }
      sync();
      for (int q = tid; q < LX * LX; q += C::NTB) {
        const int l = q / LX, i = q % LX;
#pragma unroll
        for (int tr = 0; tr < 2; ++tr) {
          const double *m = tr ? M.dxt : M.dx;
          const double a = __ldcg(m + q), mir = __ldcg(m + (N - l) * LX + (N - i));
          atomicMax(&drec[0], guard::abs_bits(a));
          atomicMax(&drec[1], guard::abs_bits(__dadd_rn(a, mir)));
        }
      }
      for (int q = tid; q < 2 * H2; q += C::NTB) {
        const int tr = q / H2, i = (q / H) % H, l = q % H;
        const double *m = tr ? M.dxt : M.dx;
        const double a = __ldcg(m + l * LX + i), b = __ldcg(m + (N - l) * LX + i);
        const df2 P = split_rn(__dmul_rn(0.5, __dadd_rn(a, b)));
        const df2 Q = split_rn(__dmul_rn(0.5, __dsub_rn(a, b)));
        cf[(tr * H + i) * CS + l] = dd2{pk(P.hi, Q.hi), pk(P.lo, Q.lo)};
        cn[tr * H2 + i * H + l] = pk(negf(P.hi), negf(Q.hi));
      }
      sync();
      const double dmax = __longlong_as_double((long long)drec[0]);
      const double ddev = __longlong_as_double((long long)drec[1]);
      raw_ok = isfinite(dmax) && ddev <= dmax * 0x1p-46;
      raw_fd = guard::d_field(drec[0]);
    } else {
      for (int q = tid; q < (int)(C::COEF_BYTES / 16); q += C::NTB)
        reinterpret_cast<ulonglong2 *>(sm)[q] =
            __ldg(reinterpret_cast<const ulonglong2 *>(M.coef) + q);
    }
  };
  // one thread: this element's geometry into Gs (completion on `bar`)
  auto issue_geo = [&](const EopPos &p) __attribute__((always_inline)) {
    const EopMesh &M = seq.mesh(seq.mesh_of(p));
    if constexpr (DROP) {  // testing aid only (a kernel of its own)
      if (seq.elem(p) == M.drop) return;
    }
    if constexpr (RAW) {
      const size_t eo = (size_t)seq.elem(p) * N3;
      const uint32_t dst = smem_u32(Gs);
      constexpr uint32_t FB = N3 * 8;
      mbar_expect(bar, 7 * FB);
      bulk_copy(dst, M.raw.g11 + eo, FB, bar);
      bulk_copy(dst + FB, M.raw.g22 + eo, FB, bar);
      bulk_copy(dst + 2 * FB, M.raw.g33 + eo, FB, bar);
      bulk_copy(dst + 3 * FB, M.raw.g12 + eo, FB, bar);
      bulk_copy(dst + 4 * FB, M.raw.g13 + eo, FB, bar);
      bulk_copy(dst + 5 * FB, M.raw.g23 + eo, FB, bar);
      bulk_copy(dst + 6 * FB, M.raw.h1 + eo, FB, bar);
    } else {
      bulk_load(smem_u32(Gs), M.gp + (size_t)seq.elem(p) * C::GE, C::GBYTES, bar);
    }
  };

  // ---- set-up: barrier, first element's geometry and inputs
  if (tid == 0) mbar_init(bar, 1);
  EopPos pos;
  bool have = seq.first(pos);
  int cmesh = -1;  // mesh whose coefficients are staged
  if constexpr (RAW) ready();
  sync();  // the barrier is initialised before anyone waits on it
  if (tid == 0 && have) issue_geo(pos);
  // one mesh: the coefficients at once, in front of ready() where they may be
  // (not with the direction update: the loop is slower so, an iteration at 26^3
  // elements, lx 10, 791 against 763 us; at lx 6, 8 and 12 within 0.5 %)
  constexpr bool kEarly = Seq::kOneMesh && !PUPD;
  if constexpr (kEarly) {
    if (have) load_coef(seq.mesh(0));
  }
  if constexpr (!RAW) ready();

  double uv[2][2] = {{0.0, 0.0}, {0.0, 0.0}};      // u (or r) of the element in turn
  double mv[2][2], pv[2][2], qv[2][2];             // PUPD: minv, old direction, corr
  auto load_in = [&](const EopPos &p) __attribute__((always_inline)) {
    const EopMesh &M = seq.mesh(seq.mesh_of(p));
    const size_t eb = (size_t)seq.elem(p) * N3;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        const size_t q = eb + pidx(b, a);
        if constexpr (PUPD) {
          uv[b][a] = up.r[q];
          mv[b][a] = up.minv[q];
          pv[b][a] = up.pw[q];
          qv[b][a] = up.corr ? up.corr[q] : 0.0;
        } else {
          uv[b][a] = __ldcg(M.u + q);
        }
      }
  };
  if (real && have) load_in(pos);

  uint32_t parity = 0;
  // outer loop: runs of elements of one mesh, whose coefficients are staged
  // before the run (measured: staging them inside the element loop, even
  // behind a test that is false after the first element, cost 6 %)
  while (have) {
    cmesh = seq.mesh_of(pos);
    if constexpr (!kEarly) load_coef(seq.mesh(cmesh));  // freed by the last barrier
  for (; have && seq.mesh_of(pos) == cmesh; parity ^= 1u) {
    EopPos nxp;
    const bool more = seq.advance(pos, nxp);
    const EopMesh &M = seq.mesh(cmesh);
    const size_t eb = (size_t)seq.elem(pos) * N3;
    // this element's admissible exponent fields of u (guard.cuh, u_range)
    const uint2 ur_e = RAW ? make_uint2(0u, 0u) : __ldcg(M.urange + seq.elem(pos));
    // ---- phase 1: this element's u (or the direction formed here), split,
    // lines of the three directions; the next element's inputs start loading
    double ucur[2][2];
    guard::Key ukk;
    double xv[2][2];
    if constexpr (PUPD && C::XUP) {
      if (real && up.x) {
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int a = 0; a < 2; ++a) xv[b][a] = up.x[eb + pidx(b, a)];
      }
    }
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        double x = uv[b][a];
        if constexpr (PUPD) {
          double z = __dmul_rn(mv[b][a], x);
          if (up.use_corr) z = __dadd_rn(z, qv[b][a]);
          x = __fma_rn(up.beta, pv[b][a], z);
          if (real) up.pw[eb + pidx(b, a)] = x;
        }
        ucur[b][a] = x;
        ukk.note(x);
      }
    df2 v[2][2];
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int a = 0; a < 2; ++a) v[b][a] = split(ucur[b][a]);
    if constexpr (PUPD && C::XUP) {
      if (real && up.x) {
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int a = 0; a < 2; ++a)
            up.x[eb + pidx(b, a)] = __fma_rn(up.alpha, pv[b][a], xv[b][a]);
      }
    }
    if (real && more) load_in(nxp);
    const unsigned uk = __reduce_max_sync(0xffffffffu, real ? ukk.get() : 0u);
    if ((tid & 31) == 0) kslot[tid >> 5] = uk;
    publish(Lb, v, v, v);
    sync();

    // ---- phase 2: reference gradient
    df2 gr[2][2], gs[2][2], gt[2][2];
    contract_all(Lb, cf, cn, gr, gs, gt);

    // ---- phase 3: pointwise h1 G with this element's staged geometry
    const bool got = mbar_wait(bar, parity, kWaitLimit);
    guard::Key gk, hk;  // RAW: exponent keys of this thread's G and h1 values
    {
      const u64 zero = pk(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        dd2 g[7];
        if constexpr (RAW) {  // fields g11, g22, g33, g12, g13, g23, h1 as staged
          const double *Gr = reinterpret_cast<const double *>(Gs);
          const int q0 = real ? pidx(b, 0) : 0, q1 = real ? pidx(b, 1) : 0;
#pragma unroll
          for (int f = 0; f < 7; ++f) {
            const double v0 = Gr[f * N3 + q0], v1 = Gr[f * N3 + q1];
            guard::Key &k = f < 6 ? gk : hk;
            k.note(v0);
            k.note(v1);
            const df2 s0 = split(v0), s1 = split(v1);
            g[f] = dd2{pk(s0.hi, s1.hi), pk(s0.lo, s1.lo)};
          }
        } else {
#pragma unroll
          for (int f = 0; f < 7; ++f) g[f] = Gs[(b * 7 + f) * NT + (real ? tid : 0)];
        }
        const dd2 UR{pk(gr[b][0].hi, gr[b][1].hi), pk(gr[b][0].lo, gr[b][1].lo)};
        const dd2 US{pk(gs[b][0].hi, gs[b][1].hi), pk(gs[b][0].lo, gs[b][1].lo)};
        const dd2 UT{pk(gt[b][0].hi, gt[b][1].hi), pk(gt[b][0].lo, gt[b][1].lo)};
        const u64 nR = neg2(UR.hi), nS = neg2(US.hi), nT = neg2(UT.hi);
        const u64 nH = neg2(g[6].hi);
        acc2 q = prod2(UR, nR, g[0]);
        mac2(q, US, nS, g[3]);
        mac2(q, UT, nT, g[4]);
        acc2 m = prod2(g[6], nH, dd2{q.s, q.c});
        gr[b][0] = df2{lx_(m.s), lx_(m.c)};
        gr[b][1] = df2{ly_(m.s), ly_(m.c)};
        q = prod2(UR, nR, g[3]);
        mac2(q, US, nS, g[1]);
        mac2(q, UT, nT, g[5]);
        m = prod2(g[6], nH, dd2{q.s, q.c});
        gs[b][0] = df2{lx_(m.s), lx_(m.c)};
        gs[b][1] = df2{ly_(m.s), ly_(m.c)};
        q = prod2(UR, nR, g[4]);
        mac2(q, US, nS, g[5]);
        mac2(q, UT, nT, g[2]);
        m = prod2(g[6], nH, dd2{q.s, q.c});
        gt[b][0] = df2{lx_(m.s), lx_(m.c)};
        gt[b][1] = df2{ly_(m.s), ly_(m.c)};
      }
    }
    if constexpr (RAW) {
      const unsigned gw = __reduce_max_sync(0xffffffffu, real ? gk.get() : 0u);
      const unsigned hw = __reduce_max_sync(0xffffffffu, real ? hk.get() : 0u);
      if ((tid & 31) == 0) {
        gslot[2 * (tid >> 5)] = gw;
        gslot[2 * (tid >> 5) + 1] = hw;
      }
    }
    // every thread is done with the geometry and the gradient lines
    if (!sync_and(got)) {
      // a staged copy never completed: record it, write NaN into this
      // group's remaining elements (so that the failure cannot pass
      // unnoticed where no status word is given) and stop (group-uniform);
      // the copy may still be in flight, so wait once more, bounded
      if (tid == 0) {
        if (err) atomicExch(err, 1);
        (void)mbar_wait(bar, parity, kWaitLimit);
      }
      for (EopPos q = pos;;) {
        double *wp = seq.mesh(seq.mesh_of(q)).w + (size_t)seq.elem(q) * N3;
        for (int i = tid; i < N3; i += C::NTB) wp[i] = __longlong_as_double(0x7ff8000000000000ll);
        EopPos q2;
        if (!seq.advance(q, q2)) break;
        q = q2;
      }
      have = false;
      break;
    }
    if (tid == 0 && more) {
      fence_async_smem();
      issue_geo(nxp);
      if constexpr (PUPD && C::XUP) {
        if (up.x) prefetch_l2(up.x + (size_t)seq.elem(nxp) * N3, N3 * 8);
      }
      if constexpr (HB) prefetch_l2(M.hb + (size_t)seq.elem(nxp) * N3, N3 * 8);
    }
    unsigned uke = 0u;
#pragma unroll
    for (int q = 0; q < NW; ++q) uke = max(uke, kslot[q]);
    bool bad;
    if constexpr (RAW) {
      unsigned gke = 0u, hke = 0u;
#pragma unroll
      for (int q = 0; q < NW; ++q) {
        gke = max(gke, gslot[2 * q]);
        hke = max(hke, gslot[2 * q + 1]);
      }
      bad = !raw_ok || !guard::window_ok(uke, gke, hke, raw_fd);
    } else {
      bad = !guard::u_in_range(ur_e, uke);
    }

    // ---- phase 4: lines of the weighted gradient
    publish(Lb, gr, gs, gt);
    sync();

    // ---- phase 5: transposed contractions, summed, stored
    contract_all(Lb, tf, tn, gr, gs, gt);
    double hv[2][2];
    if constexpr (HB) {
      if (real) {
#pragma unroll
        for (int b = 0; b < 2; ++b)
#pragma unroll
          for (int a = 0; a < 2; ++a) hv[b][a] = __ldcg(M.hb + eb + pidx(b, a));
      }
    }
    if (real && !bad) {
#pragma unroll
      for (int b = 0; b < 2; ++b) {
        dd2 acc = dsum2(dd2{pk(gr[b][0].hi, gr[b][1].hi), pk(gr[b][0].lo, gr[b][1].lo)},
                        dd2{pk(gs[b][0].hi, gs[b][1].hi), pk(gs[b][0].lo, gs[b][1].lo)});
        acc = dsum2(acc, dd2{pk(gt[b][0].hi, gt[b][1].hi), pk(gt[b][0].lo, gt[b][1].lo)});
        const df2 w0 = norm(lx_(acc.hi), lx_(acc.lo)), w1 = norm(ly_(acc.hi), ly_(acc.lo));
        double wd0 = join(w0.hi, w0.lo), wd1 = join(w1.hi, w1.lo);
        if constexpr (HB) {
          wd0 = __fma_rn(hv[b][0], ucur[b][0], wd0);
          wd1 = __fma_rn(hv[b][1], ucur[b][1], wd1);
        }
        M.w[eb + pidx(b, 0)] = wd0;
        M.w[eb + pidx(b, 1)] = wd1;
        if constexpr (DOT) {
          dsum = __fma_rn(ucur[b][0], wd0, dsum);
          dsum = __fma_rn(ucur[b][1], wd1, dsum);
        }
      }
    }
    if (bad) {  // group-uniform: fp64 units for this element
      sync();   // phase 5 has read the lines that serve as scratch
      guard::element_f64<LX>(real, M.w, PUPD ? up.pw : M.u, M.dx, M.dx, M.dx, M.dxt, M.dxt,
                             M.dxt, M.raw.h1, M.raw.g11, M.raw.g22, M.raw.g33, M.raw.g12,
                             M.raw.g13, M.raw.g23, eb, reinterpret_cast<double *>(Lb), tid, NT,
                             sync, DOT ? &dsum : nullptr);
      if constexpr (HB) {  // every thread's own points, after the barrier inside
        if (real) {
#pragma unroll
          for (int b = 0; b < 2; ++b)
#pragma unroll
            for (int a = 0; a < 2; ++a) {
              const size_t q = eb + pidx(b, a);
              M.w[q] = __fma_rn(hv[b][a], ucur[b][a], __ldcg(M.w + q));
            }
        }
      }
    }
    sync();  // the lines and key slots are free for the next element
    pos = nxp;
    have = more;
  }
  }
  if (tid == 0) {  // no copy is pending here: the barrier may be reused as plain memory
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
  }
}

// The operator handle's kernel: one mesh, elements blockIdx.x + k gridDim.x.
// DOT: one partial of u . w per CTA (fixed order) in dotp[blockIdx.x].
// DROP: the testing aid of ax_op_inject_copy_loss (plain applies only).  HB:
// with the mass term (plain applies only).
template <int LX, bool DOT, bool PUPD, bool DROP = false, bool HB = false>
__global__ void __launch_bounds__(Cfg<LX>::NTB, Cfg<LX>::MINB)
ax_eop_kernel(const EopMesh mesh, long long nelv, int *__restrict__ err,
              double *__restrict__ dotp, const EopUpd up0,
              const double *__restrict__ beta_p, const int *__restrict__ use_corr_p,
              const double *__restrict__ alpha_p) {
  using C = Cfg<LX>;
  extern __shared__ __align__(128) unsigned char sm[];
  EopUpd up = up0;
  auto ready = [&] {
    grid_wait();
    grid_go();
    if constexpr (PUPD) {  // solver scalars live on the device
      up.beta = __ldcg(beta_p);
      if constexpr (C::XUP) {
        if (up.x) up.alpha = __ldcg(alpha_p);
      }
      up.use_corr = up.corr != nullptr && __ldcg(use_corr_p) != 0;
    }
  };
  const SeqOne seq{mesh, nelv};
  double dsum = 0.0;
  eop_run<LX, DOT, PUPD, false, DROP, HB>(
      sm, (int)threadIdx.x, seq, [] { __syncthreads(); },
      [](bool p) { return __syncthreads_and(p) != 0; }, err, up, dsum, ready);
  if constexpr (DOT) {  // one partial per CTA: fixed shuffle tree, warps in order
    double *red = reinterpret_cast<double *>(sm + C::OFF_MISC + 16 + C::NW * 8);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dsum += __shfl_down_sync(0xffffffffu, dsum, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = dsum;
    __syncthreads();
    if (threadIdx.x == 0) {
      double s = 0.0;
      for (int q = 0; q < C::NW; ++q) s += red[q];
      dotp[blockIdx.x] = s;
    }
  }
}

// ax_helm on fp64 arrays: the same schedule on the caller's arrays (RAW).
template <int LX>
__global__ void __launch_bounds__(Cfg<LX>::NTB, Cfg<LX>::MINB)
ax_eopr_kernel(const EopMesh mesh, long long nelv) {
  extern __shared__ __align__(128) unsigned char sm[];
  const SeqOne seq{mesh, nelv};
  double dsum = 0.0;
  EopUpd none{};
  eop_run<LX, false, false, true>(
      sm, (int)threadIdx.x, seq, [] { __syncthreads(); },
      [](bool p) { return __syncthreads_and(p) != 0; }, nullptr, none, dsum, [] {
        grid_wait();
        grid_go();
      });
}

// Prepared geometry of this kernel: per element, entry (b * 7 + f) * NT + tid
// holds field f (g11, g22, g33, g12, g13, g23, h1) at the two points a = 0, 1
// of thread tid's corner (c, b) = (tid & 1, b), split into double-float pairs
// {hi(a=0), hi(a=1), lo(a=0), lo(a=1)} (rounded to nearest, split_rn).
// fmask picks the fields to write.
template <int LX>
__global__ void eop_prepare_kernel(df::dd2 *__restrict__ gp, const double *__restrict__ h1,
                                   const double *__restrict__ g11,
                                   const double *__restrict__ g22,
                                   const double *__restrict__ g33,
                                   const double *__restrict__ g12,
                                   const double *__restrict__ g13,
                                   const double *__restrict__ g23, int nelv, int fmask) {
  using namespace df;
  using C = Cfg<LX>;
  constexpr int H = C::H, N = C::N, H2 = C::H2, NT = C::NT, N3 = C::N3;
  const int64_t total = (int64_t)nelv * C::GE;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int tid = (int)(q % NT);
    const int f = (int)((q / NT) % 7);
    if (!((fmask >> f) & 1)) continue;
    const int b = (int)((q / (7 * NT)) % 2);
    const int64_t e = q / C::GE;
    const int t = tid >> 1, c = tid & 1;
    const int ip = t % H, jp = (t / H) % H, kp = t / H2;
    const int k = c ? N - kp : kp, j = b ? N - jp : jp;
    const double *fld = f == 0 ? g11 : f == 1 ? g22 : f == 2 ? g33 : f == 3 ? g12 : f == 4 ? g13
                      : f == 5 ? g23 : h1;
    const size_t row = (size_t)e * N3 + (size_t)(k * LX + j) * LX;
    const df2 a0 = split_rn(fld[row + ip]), a1 = split_rn(fld[row + N - ip]);
    gp[q] = dd2{pk(a0.hi, a1.hi), pk(a0.lo, a1.lo)};
  }
}

}  // namespace eop
}  // namespace ax
