// Device code of the persistent BP-SF kernel (Algorithm 1 of arXiv
// 2507.00254), included by the translation units that instantiate it
// (bpsf_inst_*.cu): one unit per kernel variant, so the instances compile in
// parallel.  The dispatch over variants and the harness kernels are in
// bpsf_kernels.cu.
//
// Execution model.  A block holds one MANAGER warp and `teams` compute teams
// of W warps.  A team decodes S work items ("slots") in lock step, one BP
// iteration at a time; a work item is the initial run of a shot (with
// oscillation counters) or one trial of a failed shot.  Per iteration a team
// runs
//   C phase : one thread per (slot, check): V2C messages times alpha, then
//             exclusion products under signed minima (Eq. c2v), C2V messages
//             written in place of the V2C messages they were computed from;
//   V phase : one thread per (slot, variable): V2C messages for the next
//             iteration (Section II-B step 2, explicit exclusion), posterior
//             LLR and hard decision (step 4), kept with the variable's flip
//             counter (Algorithm 1) in one 16-bit word; a changed decision
//             bumps the counter and toggles the slot's residual syndrome
//             s xor H e at the column's checks by shared atomics;
//   decide  : a slot whose residual syndrome is zero has converged, a slot at
//             its iteration cap is exhausted (a trial the manager found
//             unable to win under the first-success rule is stopped); the
//             slot then waits for its team's service step.
// Each message is read and written by exactly one thread in each phase, so
// one array of P floats per slot holds V2C and C2V messages alternately.
// The S slots of a team are interleaved item by item (S is a power of two):
// task tau = j*S + s (row j) or i*S + s (column i) addresses its data
// directly and a warp's lanes touch consecutive words.  A lane serves one
// slot, or 2 or 4 adjacent slots with 64- or 128-bit accesses (vector
// phases).  Installing a slot sets its messages to the channel LLRs; where
// these are all the same, the full-register instances' first C phase takes
// them as an addend instead (c_row).  With the layered schedule
// the C and V phases are replaced by layer-by-layer row updates against a
// running posterior (vector lanes for six-wide rows, else one slot per lane).
//
// Service (the team's warp 0, after an iteration in which a slot finished or
// while a slot is empty): a finished slot packs its decision into words and
// its run's facts into its outbox; a failed initial run also fills a record
// of the failure ring (Phi = top(flip_count, w), the syndrome, the shot's
// provisional output) and publishes its trials; then the slot installs the
// item the manager staged in its inbox and runs again at once.
//
// The manager warp does the rest of the global-memory work: it writes the
// outboxes out, resolves the winner of each failed shot (minimum over
// converged trials of (weight, index), merged into the shot's record by
// atomicMin), claims new shots and trials ahead of time into a small
// ready queue and fills the inboxes from it.  Compute warps touch global
// memory only when a run fails (its record) or changes a decision (the
// column's check list, in L1).
//
// Small launches, codes with ten ones per row and long codes run the column
// path (bpsf_columns.cuh) in place of the team loop.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

#include "bpsf_internal.h"

namespace bpsf {

#define FULLMASK 0xffffffffu

// Keeps a loop-invariant value in its register.  The descriptors sit in
// parameter space, indexed by the stream; left alone, the compiler loads such
// values again in every iteration (about 120 cycles for each load).
__device__ __forceinline__ int keep(int x) {
    asm volatile("" : "+r"(x));
    return x;
}
template <typename T>
__device__ __forceinline__ const T *keep(const T *p) {
    asm volatile("" : "+l"(p));
    return p;
}

__device__ __forceinline__ unsigned long long globaltimer_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long *p) {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_release_u64(unsigned long long *p, unsigned long long v) {
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ void st_release_sys_u32(volatile unsigned *p, unsigned v) {
    asm volatile("st.release.sys.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

__device__ __forceinline__ long long ld_acquire_sys_s64(const volatile long long *p) {
    long long v;
    asm volatile("ld.acquire.sys.global.s64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ unsigned long long ld_vol_u64(const unsigned long long *p) {
    return *reinterpret_cast<const volatile unsigned long long *>(p);
}

__device__ __forceinline__ unsigned ld_vol_u32(const unsigned *p) {
    return *reinterpret_cast<const volatile unsigned *>(p);
}

__device__ __forceinline__ void team_sync(int W, int bar_id) {
    if (W == 1) {
        __syncwarp();
    } else {
        asm volatile("bar.sync %0, %1;" ::"r"(bar_id), "r"(W * 32) : "memory");
    }
}

struct BlockHdr {
    int stream, cmd;
    volatile int exit;            // manager -> teams: leave the team loop
    volatile unsigned heartbeat;  // manager passes; idle teams give up only if it stalls
    unsigned long long wait_ns;   // bound on any device-side wait (column path)
    int pad[10];
};

struct LayoutMem {
    const uint8_t *row_deg;
    const uint16_t *vpos;
    const float *lch;
    const float *lch_pos;
};

struct TeamMem {
    TeamCtl *ctl;
    SlotState *st;
    uint32_t *syn, *mism, *ebits;
    unsigned char *flips;  // flip words, FB bytes each (see FlipW)
    float *m;
    OutBox *ob;         // per slot: a finished run's facts for the manager
    int *ibf;           // per slot: 1 while the inbox holds an item
    unsigned char *ib;  // per slot: the next work item
    int ibstride;
    float *post;        // layered schedule: running posterior per (variable, slot)
};

__device__ __forceinline__ TeamMem team_mem(unsigned char *tb, const TeamOffsets &to) {
    TeamMem T;
    T.ctl = reinterpret_cast<TeamCtl *>(tb + to.ctl);
    T.st = reinterpret_cast<SlotState *>(tb + to.state);
    T.syn = reinterpret_cast<uint32_t *>(tb + to.syn);
    T.mism = reinterpret_cast<uint32_t *>(tb + to.mism);
    T.ebits = reinterpret_cast<uint32_t *>(tb + to.ebits);
    T.flips = tb + to.flips;
    T.m = reinterpret_cast<float *>(tb + to.m);
    T.ob = reinterpret_cast<OutBox *>(tb + to.outbox);
    T.ibf = reinterpret_cast<int *>(tb + to.inflag);
    T.ib = tb + to.inbox;
    T.ibstride = to.ibstride;
    T.post = reinterpret_cast<float *>(tb + to.post);
    return T;
}

__device__ __forceinline__ volatile int *vstate(SlotState *s) { return reinterpret_cast<volatile int *>(&s->state); }
__device__ __forceinline__ volatile int *vflag(int *f) { return reinterpret_cast<volatile int *>(f); }

// Flip words: FB bytes per (variable, slot).  The top bit is the current hard
// decision, the bits below it count its flips (Algorithm 1): up to 32767 in
// two bytes, up to 127 in one (used only when max_iter <= 127).  Installing
// a slot zeroes them (e = 0, count 0).
template <int FB> struct FlipW;
template <> struct FlipW<2> { typedef uint16_t W; };
template <> struct FlipW<1> { typedef uint8_t W; };
template <int FB>
__device__ __forceinline__ typename FlipW<FB>::W *flipw(const TeamMem &T) {
    return reinterpret_cast<typename FlipW<FB>::W *>(T.flips);
}
template <int FB> __device__ __forceinline__ unsigned flip_dec(unsigned f) { return (f >> (8 * FB - 1)) & 1u; }
template <int FB> __device__ __forceinline__ unsigned flip_count(unsigned f) { return f & ((1u << (8 * FB - 1)) - 1u); }
// Toggle the decision and count one flip (the count is below max_iter before
// the increment, so no carry reaches the decision bit).
template <int FB> __device__ __forceinline__ unsigned flip_bump(unsigned f) { return (f ^ (1u << (8 * FB - 1))) + 1u; }

// ---------------------------------------------------------------------------
// Arithmetic of the phases.  A lane serves V adjacent slots (1, 2 or 4); two
// slots' values share one packed FP32 operation, each half rounded on its own.
// ---------------------------------------------------------------------------
template <int V> struct VecF;
template <> struct VecF<1> { typedef float T; };
template <> struct VecF<2> { typedef float2 T; };
template <> struct VecF<4> { typedef float4 T; };

template <int V>
__device__ __forceinline__ void vload(float (&x)[V], const typename VecF<V>::T *p) {
    const typename VecF<V>::T t = *p;
#pragma unroll
    for (int c = 0; c < V; ++c) x[c] = reinterpret_cast<const float *>(&t)[c];
}
template <int V>
__device__ __forceinline__ void vstore(typename VecF<V>::T *p, const float (&x)[V]) {
    typename VecF<V>::T t;
#pragma unroll
    for (int c = 0; c < V; ++c) reinterpret_cast<float *>(&t)[c] = x[c];
    *p = t;
}

// o = a * b, a + b, a - b, slot by slot.
#define BPSF_VOP(name, op, scalar)                                                                                  \
    template <int V>                                                                                                \
    __device__ __forceinline__ void name(float (&o)[V], const float (&a)[V], const float (&b)[V]) {                 \
        if (V == 1) {                                                                                               \
            o[0] = scalar(a[0], b[0]);                                                                              \
        } else {                                                                                                    \
            _Pragma("unroll") for (int c = 0; c + 1 < V; c += 2)                                                    \
                asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\t" op                     \
                    " x, x, y;\n\tmov.b64 {%0, %1}, x;\n\t}"                                                         \
                    : "=f"(o[c]), "=f"(o[c + 1])                                                                    \
                    : "f"(a[c]), "f"(a[c + 1]), "f"(b[c]), "f"(b[c + 1]));                                          \
        }                                                                                                           \
    }
BPSF_VOP(vmul, "mul.rn.f32x2", __fmul_rn)
BPSF_VOP(vadd, "add.rn.f32x2", __fadd_rn)
BPSF_VOP(vsub, "sub.rn.f32x2", __fsub_rn)
#undef BPSF_VOP

// a * b + d, slot by slot, rounded once.
template <int V>
__device__ __forceinline__ void vfma(float (&o)[V], const float (&a)[V], const float (&b)[V], const float (&d)[V]) {
    if (V == 1) {
        o[0] = __fmaf_rn(a[0], b[0], d[0]);
    } else {
#pragma unroll
        for (int c = 0; c + 1 < V; c += 2)
            asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 z, {%6, %7};\n\t"
                "fma.rn.f32x2 x, x, y, z;\n\tmov.b64 {%0, %1}, x;\n\t}"
                : "=f"(o[c]), "=f"(o[c + 1])
                : "f"(a[c]), "f"(a[c + 1]), "f"(b[c]), "f"(b[c + 1]), "f"(d[c]), "f"(d[c + 1]));
    }
}

// -(a - b), where a is not -0, slot by slot: the sign bit is set exactly when
// a > b.  b - a in its place is -0 for a = +0, b = -0, which a zero posterior
// whose last input is a zero of the other sign comes to: with one prior for all
// columns and alpha = 0.5 one [[72]] shot in eleven was decided otherwise.
template <int V>
__device__ __forceinline__ void vnegdiff(float (&o)[V], const float (&a)[V], const float (&b)[V]) {
    float zero[V];
#pragma unroll
    for (int c = 0; c < V; ++c) zero[c] = 0.f;
    vsub<V>(o, a, b);
    vsub<V>(o, zero, o);
}

// What the phases of the team path read of the code in every iteration, in registers.
struct Hot {
    int M, N, Mp;
    const uint16_t *vchk;
    bool uniform;  // all channel LLRs are lch0
    float lch0;
};

// min(|a|, |b|) with the product of the two signs: one instruction.
__device__ __forceinline__ float min_sign(float a, float b) {
    float o;
    asm("min.xorsign.abs.f32 %0, %1, %2;" : "=f"(o) : "f"(a), "f"(b));
    return o;
}
template <int V>
__device__ __forceinline__ void vmins(float (&o)[V], const float (&a)[V], const float (&b)[V]) {
#pragma unroll
    for (int c = 0; c < V; ++c) o[c] = min_sign(a[c], b[c]);
}

// ---------------------------------------------------------------------------
// Check-node update, Eq. (c2v): with a o b = (the signs' product) min(|a|, |b|),
//   out_k = seed o (o over k' != k of alpha q_k'),
// seed = 2^100 with the sign of the row's syndrome bit.  The minimum is exact
// and multiplication by alpha > 0 is monotone, so this equals alpha times the
// minimum over the other variables, clamped at 2^100, bit for bit and in any
// grouping; the sign is the XOR of the sign bits (V2C messages are never -0:
// each is a fold that starts at a channel LLR > 0, and an exact cancellation
// rounds to +0).
//
// A six-wide row takes 14 operations o for its outputs.  Keeping the two
// smallest magnitudes and selecting per output took seven ALU operations per
// edge, and the loop ran at 75 % of the ALU pipe.
// ---------------------------------------------------------------------------
// C2V magnitudes are clamped here (2^100): never reached with a fixed alpha at
// the configurations; keeps messages finite when adaptive damping tends to 1.
constexpr float kMagClamp = 0x1p100f;

// Back-off of an idle team's service loop (ns), after kIdleLooks looks that
// found nothing; the manager backs off after kIdleLooks passes without progress.
constexpr unsigned kIdleMinNs = 100, kIdleMaxNs = 2048, kIdleLooks = 16;

// Damping factor of iteration t (1-based) of a run: the fixed alpha, or the
// adaptive 1 - 2^-t (alpha == 0), an exactly rounded float subtraction
// (2^-t is exact; t >= 25 rounds to 1).
__device__ __forceinline__ float damping(const CodeDev &cd, int t) {
    const float tiny = __int_as_float((127 - min(t, 126)) << 23);
    return cd.alpha > 0.f ? cd.alpha : __fsub_rn(1.0f, tiny);
}

// Seeds of a row for V slots: syndrome bits in the low bits of sb.  NEG: the
// outputs carry the opposite sign (see the V phase).
template <int V, bool NEG>
__device__ __forceinline__ void row_seed(float (&sd)[V], unsigned sb) {
#pragma unroll
    for (int c = 0; c < V; ++c)
        sd[c] = __uint_as_float((((NEG ? ~sb : sb) << (31 - c)) & 0x80000000u) | 0x71800000u);
}

// x_k (already times alpha) -> out_k, in place; edges a row does not have hold
// +infinity (neutral).  Pairs' products, a prefix and a suffix scan over the
// pairs, then each edge takes its pair's exclusion with its partner.  Rows
// wider than eight compute the pairs' products twice rather than keep them.
template <int DC, int V>
__device__ __forceinline__ void row_outputs(float (&x)[DC][V], const float (&seed)[V]) {
    static_assert(DC % 2 == 0 && DC >= 4, "rows are padded to pairs");
    constexpr int n = DC / 2;
    constexpr bool kKeep = DC <= 8;
    float pr[kKeep ? n : 1][V], pre[n][V], run[V], e[V];
#pragma unroll
    for (int c = 0; c < V; ++c) pre[0][c] = seed[c];
#pragma unroll
    for (int i = 0; i < n; ++i) {
        float *p = pr[kKeep ? i : 0];
#pragma unroll
        for (int c = 0; c < V; ++c) {
            if (kKeep || i + 1 < n) p[c] = min_sign(x[2 * i][c], x[2 * i + 1][c]);
            if (i + 1 < n) pre[i + 1][c] = min_sign(pre[i][c], p[c]);
        }
    }
#pragma unroll
    for (int i = n - 1; i >= 0; --i) {
#pragma unroll
        for (int c = 0; c < V; ++c) {
            e[c] = i == n - 1 ? pre[i][c] : min_sign(pre[i][c], run[c]);
            if (i > 0) {
                const float p = kKeep ? pr[kKeep ? i : 0][c] : min_sign(x[2 * i][c], x[2 * i + 1][c]);
                run[c] = i == n - 1 ? p : min_sign(run[c], p);
            }
            const float o = min_sign(x[2 * i + 1][c], e[c]);
            x[2 * i + 1][c] = min_sign(x[2 * i][c], e[c]);
            x[2 * i][c] = o;
        }
    }
}

// One row for V adjacent slots.  tauv = j*(S/V) + q; MQ: rank stride in V-slot groups.
// The factors' inputs are alpha q + beta.  A running slot has its damping factor
// and -0 (which changes nothing).  In the first iteration of a run whose channel
// LLRs are all the same, alpha is 0 and beta the damped LLR: its messages need
// not be set up, which took as much shared-memory traffic as two iterations.
template <int DC, bool REG, int V>
__device__ __forceinline__ void c_row(const LayoutMem &L, const TeamMem &T, int MQ, int lgQ, int tauv,
                                      const float (&alpha)[V], const float (&beta)[V]) {
    typedef typename VecF<V>::T VT;
    VT *pv = reinterpret_cast<VT *>(T.m) + tauv;
    const int deg = REG ? DC : (int)L.row_deg[tauv >> lgQ];
    const unsigned sb = T.syn[(V * tauv) >> 5] >> ((V * tauv) & 31);
    float x[DC][V], seed[V];
#pragma unroll
    for (int k = 0; k < DC; ++k)
        if (REG || k < deg) {
            vload<V>(x[k], pv + k * MQ);
            vfma<V>(x[k], x[k], alpha, beta);
        } else {
#pragma unroll
            for (int c = 0; c < V; ++c) x[k][c] = __int_as_float(0x7f800000);
        }
    row_seed<V, true>(seed, sb);
    row_outputs<DC, V>(x, seed);
#pragma unroll
    for (int k = 0; k < DC; ++k)
        if (REG || k < deg) vstore<V>(pv + k * MQ, x[k]);
}

template <int DC, bool REG, int V>
__device__ __forceinline__ void c_phase(const Hot &h, const LayoutMem &L, const TeamMem &T, int lgS,
                                        const float (&alpha)[V], const float (&beta)[V], int tid, int nthreads) {
    const int lgQ = lgS - (V == 4 ? 2 : V - 1);
    const int MQ = h.Mp << lgQ;  // rank stride of the active layout, in V-slot groups
    const int nt = h.M << lgQ;   // row tasks (rows M..Mp-1 of the stride are padding)
    for (int tauv = tid; tauv < nt; tauv += nthreads) c_row<DC, REG, V>(L, T, MQ, lgQ, tauv, alpha, beta);
}

// ---------------------------------------------------------------------------
// V phase: variable-node update (Section II-B steps 2 and 4) and oscillation
// tracking (Algorithm 1).  For column i with C2V inputs r_0..r_{d-1} in
// ascending check order:
//   q_k   = l_ch + sum_{k' != k} r_k'   (left fold, ascending k'),
//   l_out = l_ch + sum_k r_k            (left fold),  e_i = [l_out <= 0].
// The C phase stores -r, so every step of a fold is one subtraction (the same
// rounding).  A fold starts above zero, so it is never -0 (a difference is -0
// only for -0 less +0), and 0 - l_out has its sign bit set exactly when
// l_out > 0 and is +0 for a zero (vnegdiff), so the decision is a sign bit and
// the slots' decisions are gathered by byte permutes.
//
// Lane l serves the V adjacent slots V*q .. V*q + V-1, q = l mod S/V.  Their
// items are adjacent words, so one access of up to 128 bits moves all V slots'
// messages; column tables, LLRs, addresses and loop control are shared, and
// the V slots' residual-syndrome bits of a check sit in one word.  A slot of
// the group that is not running is computed on its own stale data and its
// messages are rewritten harmlessly (an install resets them); its
// decision/flip word and syndrome bits are left alone.
// ---------------------------------------------------------------------------

// The flip words of V adjacent slots packed in one integer U (slot c in the
// c-th FB-byte field).  on: the top bits of the fields of the slots in a mask.
// diff: the top bits of the running slots' fields whose decision changes,
// given -l_out.  bump: toggle the decision and add one flip there; a count is
// below max_iter before the increment, so no carry leaves its field.  slots:
// the changed slots as a mask.
template <int FB, int V> struct FlipPack;
template <int FB> struct FlipPack<FB, 1> {
    typedef typename FlipW<FB>::W U;
    typedef unsigned D;
    static __device__ __forceinline__ D on(unsigned m) { return (m & 1u) << (8 * FB - 1); }
    static __device__ __forceinline__ D diff(const float (&nl)[1], U w, D on) {
        return (~(__float_as_uint(nl[0]) >> (32 - 8 * FB)) ^ (unsigned)w) & on;
    }
    static __device__ __forceinline__ bool any(D d) { return d != 0u; }
    static __device__ __forceinline__ U bump(U w, D d) { return (U)(((unsigned)w ^ d) + (d >> (8 * FB - 1))); }
    static __device__ __forceinline__ unsigned slots(D d) { return d >> (8 * FB - 1); }
};
__device__ __forceinline__ unsigned sign_halves(float a, float b) {
    return __byte_perm(__float_as_uint(a), __float_as_uint(b), 0xffbb);
}
template <> struct FlipPack<2, 2> {
    typedef uint32_t U;
    typedef unsigned D;
    static __device__ __forceinline__ D on(unsigned m) { return ((m & 1u) << 15) | ((m & 2u) << 30); }
    static __device__ __forceinline__ D diff(const float (&nl)[2], U w, D on) { return (~sign_halves(nl[0], nl[1]) ^ w) & on; }
    static __device__ __forceinline__ bool any(D d) { return d != 0u; }
    static __device__ __forceinline__ U bump(U w, D d) { return (w ^ d) + (d >> 15); }
    static __device__ __forceinline__ unsigned slots(D d) { return ((d >> 15) & 1u) | ((d >> 30) & 2u); }
};
template <> struct FlipPack<2, 4> {
    typedef uint2 U;
    typedef uint2 D;
    typedef FlipPack<2, 2> H;
    static __device__ __forceinline__ D on(unsigned m) { return make_uint2(H::on(m), H::on(m >> 2)); }
    static __device__ __forceinline__ D diff(const float (&nl)[4], U w, D on) {
        return make_uint2((~sign_halves(nl[0], nl[1]) ^ w.x) & on.x, (~sign_halves(nl[2], nl[3]) ^ w.y) & on.y);
    }
    static __device__ __forceinline__ bool any(D d) { return (d.x | d.y) != 0u; }
    static __device__ __forceinline__ U bump(U w, D d) { return make_uint2(H::bump(w.x, d.x), H::bump(w.y, d.y)); }
    static __device__ __forceinline__ unsigned slots(D d) { return H::slots(d.x) | (H::slots(d.y) << 2); }
};
template <> struct FlipPack<1, 2> {
    typedef uint16_t U;
    typedef unsigned D;
    static __device__ __forceinline__ D on(unsigned m) { return ((m & 1u) << 7) | ((m & 2u) << 14); }
    static __device__ __forceinline__ D diff(const float (&nl)[2], U w, D on) {
        return (~__byte_perm(__float_as_uint(nl[0]), __float_as_uint(nl[1]), 0xfbfb) ^ (unsigned)w) & on;
    }
    static __device__ __forceinline__ bool any(D d) { return d != 0u; }
    static __device__ __forceinline__ U bump(U w, D d) { return (U)(((unsigned)w ^ d) + (d >> 7)); }
    static __device__ __forceinline__ unsigned slots(D d) { return ((d >> 7) & 1u) | ((d >> 14) & 2u); }
};
template <> struct FlipPack<1, 4> {
    typedef uint32_t U;
    typedef unsigned D;
    static __device__ __forceinline__ D on(unsigned m) { return ((m * 0x00204081u) & 0x01010101u) << 7; }
    static __device__ __forceinline__ D diff(const float (&nl)[4], U w, D on) {
        const unsigned p = __byte_perm(__float_as_uint(nl[0]), __float_as_uint(nl[1]), 0xfbfb);
        const unsigned q = __byte_perm(__float_as_uint(nl[2]), __float_as_uint(nl[3]), 0xfbfb);
        return (~__byte_perm(p, q, 0x5410) ^ w) & on;
    }
    static __device__ __forceinline__ bool any(D d) { return d != 0u; }
    static __device__ __forceinline__ U bump(U w, D d) { return (w ^ d) + (d >> 7); }
    // Bits 7, 15, 23, 31 to 0..3: the four partial products meet no other in the top bits.
    static __device__ __forceinline__ unsigned slots(D d) { return ((d >> 7) * 0x10204080u) >> 28; }
};

// The residual syndrome s xor H e toggles at the checks of column i for the
// slots in bm (bit c*S + s of the team's residual-syndrome words).
template <int DVS, int DVX>
__device__ __forceinline__ void toggle_residual(const uint16_t *vchk, const TeamMem &T, int lgS, int s0, int i,
                                                unsigned bm) {
    const uint16_t *vc = vchk + i * DVS;
    uint16_t chk[DVS];
    if (DVS == 4) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2 *>(vc));
        chk[0] = (uint16_t)(raw.x & 0xffffu);
        chk[1] = (uint16_t)(raw.x >> 16);
        chk[2] = (uint16_t)(raw.y & 0xffffu);
        chk[3] = (uint16_t)(raw.y >> 16);
    } else {
#pragma unroll
        for (int k = 0; k < DVS; ++k) chk[k] = __ldg(vc + k);
    }
#pragma unroll
    for (int k = 0; k < DVS; ++k) {
        if (DVX > 0 ? (k < DVX) : (chk[k] != 0xffffu)) {
            const int b = ((int)chk[k] << lgS) + s0;
            atomicXor(&T.mism[b >> 5], bm << (b & 31));
        }
    }
}

template <int DVS, int DVX, bool DEBUG, int V, int FB, bool UNI>
__device__ __forceinline__ void v_phase(const StreamDev &sd, const Hot &h, const LayoutMem &L, const TeamMem &T, int lgS,
                                        unsigned onm, unsigned initm, int tid, int nthreads) {
    typedef typename VecF<V>::T VT;
    typedef FlipPack<FB, V> FP;
    const int lgQ = lgS - (V == 4 ? 2 : V - 1);
    const int total = h.N << lgQ;
    const int q = tid & ((1 << lgQ) - 1);
    const int s0 = V * q;
    VT *mv = reinterpret_cast<VT *>(T.m) + q;
    typename FP::U *fv = reinterpret_cast<typename FP::U *>(T.flips);
    const typename FP::D on = FP::on(onm);
    constexpr int DV = DVX > 0 ? DVX : DVS;  // entries looked at (the rest of the table is padding)
    for (int tauv = tid; tauv < total; tauv += nthreads) {
        const int i = tauv >> lgQ;
        uint16_t pos[DVS];
        const uint16_t *vp = L.vpos + i * DVS;
        if (DVS == 4) {
            const uint2 raw = *reinterpret_cast<const uint2 *>(vp);
            pos[0] = (uint16_t)(raw.x & 0xffffu);
            pos[1] = (uint16_t)(raw.x >> 16);
            pos[2] = (uint16_t)(raw.y & 0xffffu);
            pos[3] = (uint16_t)(raw.y >> 16);
        } else {
#pragma unroll
            for (int k = 0; k < DVS; ++k) pos[k] = vp[k];
        }
        float lc[V];
        {
            const float l = UNI && h.uniform ? h.lch0 : L.lch[i];
#pragma unroll
            for (int c = 0; c < V; ++c) lc[c] = l;
        }
        // A missing entry reads as 0: subtracting +0 changes nothing.
        float r[DV][V];
#pragma unroll
        for (int k = 0; k < DV; ++k) {
            if (DVX > 0 || pos[k] != 0xffffu) {
                vload<V>(r[k], mv + ((int)pos[k] << lgQ));
            } else {
#pragma unroll
                for (int c = 0; c < V; ++c) r[k][c] = 0.f;
            }
        }
        const typename FP::U fw = fv[tauv];
        // pre = l_ch + r_0 + .. + r_{k-1}; q_k goes on from there without r_k.
        float pre[V], nl[V];
#pragma unroll
        for (int c = 0; c < V; ++c) pre[c] = lc[c];
#pragma unroll
        for (int k = 0; k < DV; ++k) {
            float acc[V];
#pragma unroll
            for (int c = 0; c < V; ++c) acc[c] = pre[c];
#pragma unroll
            for (int k2 = k + 1; k2 < DV; ++k2) vsub<V>(acc, acc, r[k2]);
            if (k + 1 < DV)
                vsub<V>(pre, pre, r[k]);
            else
                vnegdiff<V>(nl, pre, r[k]);  // -l_out
            if (DVX > 0 || pos[k] != 0xffffu) vstore<V>(mv + ((int)pos[k] << lgQ), acc);
        }
        if (DEBUG && sd.dbg.lout) {
#pragma unroll
            for (int c = 0; c < V; ++c)
                if (((onm >> c) & 1u) && ((initm >> (s0 + c)) & 1u))
                    sd.dbg.lout[T.st[s0 + c].shot * h.N + i] = __fsub_rn(0.f, nl[c]);
        }
        const typename FP::D d = FP::diff(nl, fw, on);
        if (FP::any(d)) {
            fv[tauv] = FP::bump(fw, d);
            toggle_residual<DVS, DVX>(h.vchk, T, lgS, s0, i, FP::slots(d));
        }
    }
}

// ---------------------------------------------------------------------------
// Layered schedule.  Layer by layer (rows of a layer share no variable, so
// they run in parallel and in any order), each row j of slot s:
// q_k = L_i - r_k for its edges k (i = the k-th variable of the row, r_k its
// C2V message from the previous iteration), new C2V messages from the q_k by
// Eq. (c2v) as in the C phase, then L_i = q_k + r_k.  After all layers L is the
// posterior: hard decision, flip counters and residual syndrome as in the V
// phase.  A lane serves V adjacent slots; slots of the group that are not
// running compute on stale values, and their results are never read (a slot's
// messages and posterior are set up again when it takes its next item).
// ---------------------------------------------------------------------------
template <int DC, bool REG, int V>
__device__ __forceinline__ void layered_row(const CodeDev &cd, const LayoutMem &L, const TeamMem &T, int lgQ, int j,
                                            int q, const float (&alpha)[V]) {
    typedef typename VecF<V>::T VT;
    const int M = cd.Mp, MQ = cd.Mp << lgQ;  // rank stride of the active layout (in V-slot groups: MQ)
    const int deg = REG ? DC : (int)L.row_deg[j];
    VT *mj = reinterpret_cast<VT *>(T.m) + (j << lgQ) + q;  // edge k of row j at (k*M + j)*Q + q
    VT *pv = reinterpret_cast<VT *>(T.post) + q;            // posterior of variable i at i*Q + q
    float qv[DC][V], x[DC][V], seed[V];
#pragma unroll
    for (int k = 0; k < DC; ++k) {
        if (REG || k < deg) {
            float lp[V], r[V];
            vload<V>(lp, pv + ((int)__ldg(cd.pos_var + k * M + j) << lgQ));
            vload<V>(r, mj + k * MQ);
            vsub<V>(qv[k], lp, r);
            vmul<V>(x[k], qv[k], alpha);
        } else {
#pragma unroll
            for (int c = 0; c < V; ++c) x[k][c] = __int_as_float(0x7f800000);
        }
    }
    const int b0 = V * ((j << lgQ) + q);  // syndrome bit of row j, first slot of the group
    row_seed<V, false>(seed, T.syn[b0 >> 5] >> (b0 & 31));
    row_outputs<DC, V>(x, seed);
#pragma unroll
    for (int k = 0; k < DC; ++k) {
        if (REG || k < deg) {
            float np[V];
            vadd<V>(np, qv[k], x[k]);
            vstore<V>(mj + k * MQ, x[k]);
            vstore<V>(pv + ((int)__ldg(cd.pos_var + k * M + j) << lgQ), np);  // read again: fewer live registers
        }
    }
}

template <int DC, int DVS, int DVX, bool DEBUG, int V, int FB>
__device__ __forceinline__ void layered_iteration(const StreamDev &sd, const LayoutMem &L, const TeamMem &T, int lgS,
                                                  unsigned onm, const float (&alpha)[V], unsigned initm, int tid,
                                                  int nthreads, int W, int bar_id) {
    typedef typename VecF<V>::T VT;
    typedef FlipPack<FB, V> FP;
    const CodeDev &cd = sd.code;
    const int lgQ = lgS - (V == 4 ? 2 : V - 1);
    const int q = tid & ((1 << lgQ) - 1);  // the lane's slot group: slots V*q .. V*q + V-1
    const int s0 = V * q;
    for (int layer = 0; layer < cd.n_layers; ++layer) {
        const int r0 = (int)__ldg(cd.layer_ptr + layer), r1 = (int)__ldg(cd.layer_ptr + layer + 1);
        const int total = (r1 - r0) << lgQ;
        if (onm)
            for (int tauv = tid; tauv < total; tauv += nthreads)
                layered_row<DC, (DVX > 0), V>(cd, L, T, lgQ, (int)__ldg(cd.layer_rows + r0 + (tauv >> lgQ)), q, alpha);
        team_sync(W, bar_id);
    }
    if (!onm) return;
    const int N = cd.N;
    const VT *pv = reinterpret_cast<const VT *>(T.post);
    typename FP::U *fv = reinterpret_cast<typename FP::U *>(T.flips);
    const typename FP::D on = FP::on(onm);
    for (int tauv = tid; tauv < (N << lgQ); tauv += nthreads) {
        const int i = tauv >> lgQ;
        float lo[V], nl[V];
        vload<V>(lo, pv + tauv);
        const typename FP::U fw = fv[tauv];
#pragma unroll
        for (int c = 0; c < V; ++c) {
            nl[c] = __fsub_rn(0.f, lo[c]);  // a zero of either sign comes out as +0: decided 1
            if (DEBUG && sd.dbg.lout && ((onm >> c) & 1u) && ((initm >> (s0 + c)) & 1u))
                sd.dbg.lout[T.st[s0 + c].shot * N + i] = lo[c];
        }
        const typename FP::D d = FP::diff(nl, fw, on);
        if (FP::any(d)) {
            fv[tauv] = FP::bump(fw, d);
            toggle_residual<DVS, DVX>(cd.vchk, T, lgS, s0, i, FP::slots(d));
        }
    }
}

// ---------------------------------------------------------------------------
// Team-side slot service (warp 0 of the team, all lanes).  A finished slot
// (PENDING) hands its facts to its outbox as soon as the manager has drained
// the previous ones; a free slot (EMPTY) installs the item the manager put
// in its inbox.  The slot therefore runs again at the team's next iteration,
// without a round trip through the manager.
// ---------------------------------------------------------------------------

// The record of slot s's failed initial run: Phi = top(flip_count, w) (keys
// (count << 16 | 0xffff - i) are distinct, so each round takes the largest
// key below the previous one: count descending, index ascending), the shot's
// syndrome, an empty selection and the provisional output (the initial run's
// e, not converged); only then is the record published for the trials.
// Called by one warp, with the slot's flip words and packed decision in place.
template <bool DEBUG, int FB, bool COLS>
__device__ __forceinline__ void publish_failure(const StreamDev &sd, const TeamMem &T, int lgS, int s, int lane,
                                                unsigned long long wait_ns) {
    const CodeDev &cd = sd.code;
    const int N = cd.N, Wn = cd.Wn;
    const JobDev &job = sd.job;
    const long long shot = T.st[s].shot;
    const long long row = (sd.flags & kServe) ? (shot % sd.serve.rows) : shot;
    // Phi into lane registers: lane r % 32 holds Phi[r] (r < 32 in phi0, else phi1).
    int phi0 = -1, phi1 = -1;
    unsigned thr = 0xffffffffu;
    for (int r = 0; r < cd.w; ++r) {
        unsigned best = 0;
        for (int i = lane; i < N; i += 32) {
            const unsigned key =
                (flip_count<FB>((unsigned)flipw<FB>(T)[(i << lgS) + s]) << 16) | (0xffffu - (unsigned)i);
            if (key < thr && key > best) best = key;
        }
        best = __reduce_max_sync(FULLMASK, best);
        const int phi_r = (int)(0xffffu - (best & 0xffffu));
        if (lane == (r & 31)) {
            if (r < 32)
                phi0 = phi_r;
            else
                phi1 = phi_r;
        }
        if (DEBUG && lane == 0 && sd.dbg.phi) sd.dbg.phi[shot * cd.w + r] = phi_r;
        thr = best;
    }
    // The next failure number and its record, once free (a bounded wait;
    // more failed shots in flight than records is reported).
    unsigned long long q = 0;
    if (lane == 0) {
        q = atomicAdd(&sd.ctr->rec_count, 1ull);
        const unsigned long long *qs = sd.rec.qseq + (q & (unsigned long long)(sd.rec.cap - 1));
        auto busy = [&] {
            const unsigned long long v = ld_acquire_u64(qs);
            return v != 0ull && !(v & kRecFree);
        };
        if (busy()) {
            const unsigned long long t0 = globaltimer_ns();
            while (busy()) {
                if (globaltimer_ns() - t0 > wait_ns) {
                    atomicOr(&sd.ctr->status, kDevRecordOverflow);
                    break;
                }
                __nanosleep(256);
            }
        }
    }
    q = __shfl_sync(FULLMASK, q, 0);
    const long long rs = (long long)(q & (unsigned long long)(sd.rec.cap - 1));
    if (lane < cd.w) sd.rec.phi[rs * cd.w + lane] = phi0;
    if (lane + 32 < cd.w) sd.rec.phi[rs * cd.w + lane + 32] = phi1;
    // The slot's syndrome: its own words (COLS), or bit j*S + s of the team's words for check j.
    if (COLS) {
        for (int w = lane; w < cd.Ws; w += 32) sd.rec.synd[rs * cd.Ws + w] = T.syn[s * cd.Ws + w];
    } else {
        for (int w = 0; w < cd.Ws; ++w) {
            const int j = 32 * w + lane;
            const int b = (j << lgS) + s;
            const unsigned bit = j < cd.M ? (T.syn[b >> 5] >> (b & 31)) & 1u : 0u;
            const unsigned word = __ballot_sync(FULLMASK, bit != 0u);
            if (lane == 0) sd.rec.synd[rs * cd.Ws + w] = word;
        }
    }
    __syncwarp();  // lane 0's decision words are visible to the warp
    uint32_t *out = job.corr + row * job.corr_stride;
    for (int w = lane; w < Wn; w += 32) {
        sd.rec.win[rs * Wn + w] = ~0ull;
        out[w] = T.ebits[s * Wn + w];
    }
    if (lane == 0) {
        job.conv[row] = 0;
        job.iters[row] = (int16_t)cd.max_iter;
        if (job.stage) job.stage[row] = 2;
        sd.rec.done[rs] = 0u;
        sd.rec.best[rs] = ~0ull;
        sd.rec.qshot[rs] = shot;
    }
    __threadfence();
    __syncwarp();
    if (lane == 0) st_release_u64(sd.rec.qseq + rs, q + 1ull);
}

// Pack finished slot s into its outbox: the hard decision into words and the
// run's facts.  A failed initial run (with trials) also gets its record here.
template <bool DEBUG, int FB>
__device__ __forceinline__ void team_pack(const StreamDev &sd, const TeamMem &T, int lgS, int s, int lane,
                                          unsigned long long wait_ns) {
    const CodeDev &cd = sd.code;
    const int N = cd.N, Wn = cd.Wn;
    const SlotState *ss = &T.st[s];
    OutBox *ob = &T.ob[s];
    for (int w = 0; w < Wn; ++w) {
        const int i = 32 * w + lane;
        const unsigned b = i < N ? flip_dec<FB>((unsigned)flipw<FB>(T)[(i << lgS) + s]) : 0u;
        const unsigned word = __ballot_sync(FULLMASK, b != 0u);
        if (lane == 0) T.ebits[s * Wn + w] = word;
    }
    const int kind = ss->kind, outcome = ss->outcome;
    if (kind == 1 && outcome == 2 && cd.w > 0) publish_failure<DEBUG, FB, false>(sd, T, lgS, s, lane, wait_ns);
    if (DEBUG && kind == 1 && sd.dbg.flips)
        for (int i = lane; i < N; i += 32)
            sd.dbg.flips[ss->shot * N + i] = (uint16_t)flip_count<FB>((unsigned)flipw<FB>(T)[(i << lgS) + s]);
    if (lane == 0) {
        ob->kind = kind;
        ob->kidx = ss->kidx;
        ob->rec = ss->rec;
        ob->outcome = outcome;
        ob->iter = ss->iter;
        ob->shot = ss->shot;
    }
    __syncwarp();
    if (lane == 0) {
        __threadfence_block();
        *vflag(&ob->full) = 1;
    }
    __syncwarp();
}

// Install slot s's inbox item: the slot's bits of the syndrome and
// residual-syndrome words (atomic toggles of the bits that differ: lanes
// share words), its V2C messages set to the channel LLRs (the first C phase
// reads l_ch on every edge), its decision and flip-count words zeroed.
template <int FB, bool UNI>
__device__ __forceinline__ void team_install(const StreamDev &sd, const LayoutMem &L, const TeamMem &T, int S, int s,
                                             int lane) {
    const CodeDev &cd = sd.code;
    const QEntry *e = reinterpret_cast<const QEntry *>(T.ib + s * T.ibstride);
    const uint32_t *src = reinterpret_cast<const uint32_t *>(T.ib + s * T.ibstride + sizeof(QEntry));
    SlotState *ss = &T.st[s];
    volatile uint32_t *vsyn = T.syn, *vmism = T.mism;
    for (int j = lane; j < cd.M; j += 32) {
        const unsigned want = (src[j >> 5] >> (j & 31)) & 1u;
        const int b = j * S + s;
        const unsigned m = 1u << (b & 31);
        if (((vsyn[b >> 5] & m) != 0u) != (want != 0u)) atomicXor(&T.syn[b >> 5], m);
        if (((vmism[b >> 5] & m) != 0u) != (want != 0u)) atomicXor(&T.mism[b >> 5], m);
    }
    if (cd.layered) {
        // Layered schedule: C2V messages start at zero, the posterior at l_ch.
        for (int k = lane; k < cd.P; k += 32) T.m[k * S + s] = 0.f;
        for (int i = lane; i < cd.N; i += 32) T.post[i * S + s] = L.lch[i];
    } else if (!UNI || !cd.uniform) {  // else see c_row
        for (int k = lane; k < cd.P; k += 32) T.m[k * S + s] = L.lch_pos[k];
    }
    for (int i = lane; i < cd.N; i += 32) flipw<FB>(T)[i * S + s] = 0;
    if (lane == 0) {
        ss->kind = e->kind;
        ss->kidx = e->kidx;
        ss->rec = e->rec;
        ss->shot = e->shot;
        ss->iter = 0;
        ss->start = -1;  // set by the team at the service that starts the run
        ss->outcome = 0;
        ss->cancel = 0;
        ss->limit = e->kind == 1 ? cd.max_iter : cd.short_iter;
    }
    __syncwarp();
}

template <bool DEBUG, int FB, bool UNI>
__device__ __forceinline__ void team_service(const StreamDev &sd, const LayoutMem &L, const TeamMem &T, int S, int lgS,
                                             int lane, unsigned long long wait_ns) {
    const int stv = lane < S ? *vstate(&T.st[lane]) : kSlotRunning;
    const bool obf = lane < S && *vflag(&T.ob[lane].full) != 0;
    unsigned pm = __ballot_sync(FULLMASK, stv == kSlotPending && !obf);
    if (pm) __threadfence_block();  // the manager's reads of the drained outboxes are done
    while (pm) {
        const int s = __ffs(pm) - 1;
        pm &= pm - 1u;
        team_pack<DEBUG, FB>(sd, T, lgS, s, lane, wait_ns);
        // team_pack set the outbox flag before the slot reads EMPTY (the
        // manager's exit test reads the state first, then the outbox flag).
        if (lane == 0) {
            __threadfence_block();
            *vstate(&T.st[s]) = kSlotEmpty;
        }
    }
    __syncwarp();
    const bool want = lane < S && *vstate(&T.st[lane]) == kSlotEmpty && *vflag(&T.ibf[lane]) != 0;
    unsigned im = __ballot_sync(FULLMASK, want);
    if (im) __threadfence_block();  // the inbox items are visible
    while (im) {
        const int s = __ffs(im) - 1;
        im &= im - 1u;
        const int kind = reinterpret_cast<const QEntry *>(T.ib + s * T.ibstride)->kind;
        if (kind != 0) team_install<FB, UNI>(sd, L, T, S, s, lane);
        __syncwarp();
        if (lane == 0) {
            // RUNNING before the inbox reads empty: the manager's exit test
            // reads the inbox flag first, then the state.
            __threadfence_block();
            if (kind != 0) *vstate(&T.st[s]) = kSlotRunning;
            __threadfence_block();
            *vflag(&T.ibf[s]) = 0;
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------------------
// Compute team loop.
//
// A team iteration is: C phase, barrier, V phase, barrier, decision.  The
// decision needs no further barrier: every warp reads the residual-syndrome
// words (stable until the next V phase, which lies beyond the next barrier)
// and the iteration's stop mask (written by warp 0 before the first barrier,
// one word per iteration parity), so all warps agree on which slots are done.
// The service step (a barrier, warp 0 packs finished slots and installs new
// items, a barrier) runs only after an iteration in which a slot finished, or
// while a slot is empty, and with an iteration chunk k > 1 at most every k
// iterations while some slot still runs; a team whose slots all keep running
// goes from one iteration to the next with two barriers.
// ---------------------------------------------------------------------------
template <int DC, int DVS, int DVX, bool DEBUG, int MINB, bool LAY, int FB>
__device__ void team_loop(const StreamDev &sd, const LayoutMem &L, const TeamMem &T, BlockHdr *hdr, int S, int W,
                          int tid, int bar_id, unsigned long long wait_ns) {
    const int lane = tid & 31, wt = tid >> 5, nthreads = 32 * W;
    const CodeDev &cd = sd.code;
    const int lgS = __ffs(S) - 1;
    const int n_rwords = MINB == 1 ? keep(((cd.M << lgS) + 31) >> 5) : ((cd.M << lgS) + 31) >> 5;  // residual-syndrome words of the team
    const unsigned full = S >= 32 ? 0xffffffffu : ((1u << S) - 1u);
    constexpr bool kVec = DC <= 16;  // the widest rows keep one slot per lane (registers)
    // Four slots per lane: exact-degree rows with the full register budget (one block).
    constexpr bool kVec4 = kVec && MINB == 1 && DVX == 3;
    // Layered schedule: vector lanes in the full-register instances only.
    constexpr bool kLayV2 = LAY && kVec && MINB == 1 && DC <= 6, kLayV4 = kLayV2 && kVec4;
    const bool lay = LAY && cd.layered;
    // Not in the 64-register instance: it spills 32 B a thread as it is, and with
    // this 200 000 [[72]] shots took 6.6 instead of 5.7 ms.
    Hot h = {cd.M, cd.N, cd.Mp, cd.vchk, false, 0.f};
    if (MINB == 1) h = {keep(h.M), keep(h.N), keep(h.Mp), keep(h.vchk), keep(cd.uniform) != 0 && !lay, cd.lch0};
    const float alpha0 = cd.alpha;
    unsigned fresh = 0u;  // slots in the first iteration of their run
    // Slots per lane in the phases (vs) and the lane's first slot (s0).
    const int vs = lay ? ((kLayV4 && S >= 4) ? 4 : ((kLayV2 && S >= 2) ? 2 : 1))
                       : ((kVec4 && S >= 4) ? 4 : ((kVec && S >= 2) ? 2 : 1));
    const int s0 = vs * (lane & ((S / vs) - 1));
    unsigned run = 0u, initm = 0u;
    int tt = 0;  // team iterations run (the same in every warp)
    // Every warp, lane l < S: the team iteration after which slot l's run
    // reaches its iteration cap.
    int l_end = 0;
    // Warp 0, lane 0: iterations run since the last service, and the team
    // iteration of that service (added to the control block at the next one).
    unsigned n_iters = 0;
    int tt_flush = 0;
    const bool first_rule = cd.select == 1;
    const bool adaptive = !(cd.alpha > 0.f);  // alpha_t = 1 - 2^-t needs each run's iteration number
    bool svc = true;
    const int chunk = sd.chunk > 1 ? sd.chunk : 1;  // iterations between refills of finished slots
    int since = 0;                                  // team iterations since the last service
    // The idle state (warp 0 only, rarely used) lives in the control block.
    if (wt == 0 && lane == 0) {
        T.ctl->idle_since = 0;
        T.ctl->idle_ns = kIdleMinNs;
        T.ctl->idle_looks = 0;
    }
    for (;;) {
        if (svc) {
            // Every warp has made the previous decision (read the residual
            // words, which an install rewrites) and has read the control
            // block of the previous service.
            team_sync(W, bar_id);
            if (wt == 0) {
                // The work counters first: the manager adds them up once every
                // slot of the block reads empty, which the service below may make so.
                if (lane == 0 && tt != tt_flush) {
                    T.ctl->iters += n_iters;
                    T.ctl->cap += (unsigned long long)(tt - tt_flush) * (unsigned)S;
                    n_iters = 0;
                    tt_flush = tt;
                }
                team_service<DEBUG, FB, MINB == 1>(sd, L, T, S, lgS, lane, wait_ns);
                SlotState *ss = &T.st[lane < S ? lane : 0];
                const int stv = lane < S ? *vstate(ss) : kSlotEmpty;
                const bool r = stv == kSlotRunning;
                __threadfence_block();
                const unsigned rm = __ballot_sync(FULLMASK, r);
                const unsigned im = __ballot_sync(FULLMASK, r && ss->kind == 1);
                const unsigned fm = __ballot_sync(FULLMASK, r && ss->start < 0);
                // A run installed at this service starts with the next iteration.
                if (r && ss->start < 0) ss->start = tt;
                int ex = 0;
                if (rm == 0u) {
                    if (hdr->exit) {
                        ex = 1;
                    } else {
                        // Never wait forever: give up only if the manager has made
                        // no pass for twice the bound on any of its own waits.
                        const unsigned long long now = globaltimer_ns();
                        const unsigned beat = hdr->heartbeat;
                        unsigned long long since_ns = T.ctl->idle_since;
                        if (since_ns == 0 || beat != T.ctl->last_beat) since_ns = now;
                        if (now - since_ns > 2 * wait_ns) ex = 1;
                        // A team idle for more than a few looks backs off (up
                        // to 2 us), so the warps of the block that do run keep
                        // the issue slots; short gaps between runs keep the
                        // short sleep.
                        unsigned ns = T.ctl->idle_ns;
                        const unsigned looks = T.ctl->idle_looks + 1;
                        __nanosleep(ns);
                        if (looks > kIdleLooks) ns = ns < kIdleMaxNs ? 2 * ns : kIdleMaxNs;
                        __syncwarp();
                        if (lane == 0) {
                            T.ctl->idle_since = since_ns;
                            T.ctl->last_beat = beat;
                            T.ctl->idle_ns = ns;
                            T.ctl->idle_looks = looks;
                        }
                    }
                } else if (lane == 0) {
                    T.ctl->idle_since = 0;
                    T.ctl->idle_ns = kIdleMinNs;
                    T.ctl->idle_looks = 0;
                }
                if (lane == 0) {
                    T.ctl->run_mask = rm;
                    T.ctl->init_mask = im;
                    T.ctl->fresh = fm;
                    T.ctl->exit = ex;
                }
            }
            team_sync(W, bar_id);
            run = T.ctl->run_mask;
            initm = T.ctl->init_mask;
            if (MINB == 1) fresh = T.ctl->fresh;
            const int ex = T.ctl->exit;
            if (ex) break;
            if (run == 0u) continue;
            if (lane < S) l_end = T.st[lane].start + T.st[lane].limit - 1;
            svc = false;
            since = 0;
        }
        // First-success rule: warp 0 publishes the trials the manager asked to
        // stop (they cannot win), read by every warp after this iteration.
        if (first_rule && wt == 0) {
            bool cancel = false;
            if (lane < S && ((run >> lane) & 1u) && T.st[lane].kind == 2)
                cancel = *reinterpret_cast<volatile long long *>(&T.st[lane].cancel) ==
                         T.st[lane].shot * (long long)cd.n_trials + T.st[lane].kidx + 1;
            const unsigned cm = __ballot_sync(FULLMASK, cancel);
            if (lane == 0) T.ctl->stop_mask[tt & 1] = cm;
        }
        // Damping of iteration it = tt - start + 1 of each of the lane's slots
        // (the start is read only under adaptive damping).
        float al[4], be[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            al[c] = adaptive && c < vs ? damping(cd, tt - T.st[s0 + c].start + 1) : alpha0;
            const bool f = MINB == 1 && h.uniform && ((fresh >> (s0 + c)) & 1u) && c < vs;
            be[c] = f ? __fmul_rn(damping(cd, 1), h.lch0) : -0.0f;
            al[c] = f ? 0.f : al[c];
        }
        fresh = 0u;
        const unsigned onm = (run >> s0) & ((1u << vs) - 1u);  // the lane's running slots
        if (lay) {
            if (kLayV4 && vs == 4) {
                layered_iteration<DC, DVS, DVX, DEBUG, 4, FB>(sd, L, T, lgS, onm, al, initm, tid, nthreads, W, bar_id);
            } else if (kLayV2 && vs == 2) {
                const float a2[2] = {al[0], al[1]};
                layered_iteration<DC, DVS, DVX, DEBUG, 2, FB>(sd, L, T, lgS, onm, a2, initm, tid, nthreads, W, bar_id);
            } else {
                const float a1[1] = {al[0]};
                layered_iteration<DC, DVS, DVX, DEBUG, 1, FB>(sd, L, T, lgS, onm, a1, initm, tid, nthreads, W, bar_id);
            }
        } else if (kVec4 && vs == 4) {
            if (onm) c_phase<DC, (DVX > 0), 4>(h, L, T, lgS, al, be, tid, nthreads);
            team_sync(W, bar_id);
            if (onm) v_phase<DVS, DVX, DEBUG, 4, FB, MINB == 1>(sd, h, L, T, lgS, onm, initm, tid, nthreads);
        } else if (kVec && vs == 2) {
            const float a2[2] = {al[0], al[1]}, b2[2] = {be[0], be[1]};
            if (onm) c_phase<DC, (DVX > 0), 2>(h, L, T, lgS, a2, b2, tid, nthreads);
            team_sync(W, bar_id);
            if (onm) v_phase<DVS, DVX, DEBUG, 2, FB, MINB == 1>(sd, h, L, T, lgS, onm, initm, tid, nthreads);
        } else {
            const float a1[1] = {al[0]}, b1[1] = {be[0]};
            if (onm) c_phase<DC, (DVX > 0), 1>(h, L, T, lgS, a1, b1, tid, nthreads);
            team_sync(W, bar_id);
            if (onm) v_phase<DVS, DVX, DEBUG, 1, FB, MINB == 1>(sd, h, L, T, lgS, onm, initm, tid, nthreads);
        }
        team_sync(W, bar_id);
        // Decision, in every warp: slot s owns bits s, s + S, s + 2S, ... of
        // every residual-syndrome word, so OR-folding the words down to S
        // bits leaves bit s set iff slot s's residual syndrome is not zero.
        unsigned acc = 0;
        for (int w = lane; w < n_rwords; w += 32) acc |= T.mism[w];
        acc = __reduce_or_sync(FULLMASK, acc);
        for (int sh = 16; sh >= S; sh >>= 1) acc |= acc >> sh;
        const unsigned nconv = acc & full;
        // Runs at their iteration cap (every warp knows every slot's cap), and
        // trials asked to stop.
        const unsigned capped = __ballot_sync(FULLMASK, lane < S && tt >= l_end);
        const unsigned cancelled = first_rule ? T.ctl->stop_mask[tt & 1] : 0u;
        const unsigned done = run & (~nconv | capped | cancelled);
        if (wt == 0) {
            if ((done >> lane) & 1u) {
                SlotState *ss = &T.st[lane];
                ss->iter = tt - ss->start + 1;
                ss->outcome = !((nconv >> lane) & 1u) ? 1 : (((cancelled >> lane) & 1u) ? 3 : 2);
                // Finished slots are packed by the next service step.
                *vstate(ss) = kSlotPending;
            }
            n_iters += __popc(run);
        }
        // Finished slots leave the run mask at once (their decisions and flip
        // counts stay as they were) and wait for the next service, which comes
        // after the iteration chunk, or at once when no slot is left running.
        ++tt;
        ++since;
        run &= ~done;
        svc = run == 0u || (since >= chunk && run != full);
    }
}

// The output row of a shot.
__device__ __forceinline__ long long row_of(const StreamDev &sd, long long shot) {
    return (sd.flags & kServe) ? (shot % sd.serve.rows) : shot;
}

}  // namespace bpsf

#include "bpsf_columns.cuh"

namespace bpsf {

// ---------------------------------------------------------------------------
// Manager warp.
// ---------------------------------------------------------------------------

// Manager state: head and tail are warp-uniform; the two counters are per
// lane (each lane counts the slots it wrote out) and are summed over the
// warp before they are added to the global counters.
struct MgrState {
    int head, tail;          // ready queue (ring of Q entries)
    unsigned init_local;     // finished initial runs not yet counted globally
    unsigned trials_local;   // finished trial runs not yet counted globally
    unsigned trials_cancelled; // trials not run or stopped because they could not win
    unsigned long long stall_q, stall_since;  // a record announced, not yet written (number + 1; 0: none), and since when
};

__device__ __forceinline__ QEntry *qentry(unsigned char *q, int idx, int stride) {
    return reinterpret_cast<QEntry *>(q + idx * stride);
}

__device__ __forceinline__ uint32_t *qsyn(QEntry *e) {
    return reinterpret_cast<uint32_t *>(reinterpret_cast<unsigned char *>(e) + sizeof(QEntry));
}

// Word w of finished slot s's hard decision (packed by its team).
__device__ __forceinline__ unsigned slot_word(const uint32_t *ebits, int Wn, int s, int w) { return ebits[s * Wn + w]; }



// One shot's final output is out: when serving, post it to the row's
// completion word (the outputs live in host-mapped memory, hence the
// system-scope fence before the release).
__device__ __forceinline__ void shot_complete(const StreamDev &sd, long long row, long long shot) {
    if (!(sd.flags & kServe)) return;
    __threadfence_system();
    st_release_sys_u32(sd.serve.row_done + row, (unsigned)(shot + 1));
}

// One trial of a failed shot is over (run, or cancelled because it cannot
// win): count it; the last one settles the winner (the minimum key of the
// shot's converged trials) and completes the shot.
template <bool COLS>
__device__ __forceinline__ void trial_done(const StreamDev &sd, long long rs, long long row, long long shot,
                                           bool merged) {
    const CodeDev &cd = sd.code;
    const JobDev &job = sd.job;
    const int C = cd.n_trials, Wn = cd.Wn;
    if (merged) __threadfence();  // its words before its count
    const unsigned d = (atomicAdd(&sd.rec.done[rs], 1u) + 1u) & ((1u << kDoneBits) - 1u);
    if (d == (unsigned)C) {
        __threadfence();
        const unsigned long long best = atomicAdd(&sd.rec.best[rs], 0ull);
        if (best != ~0ull) {
            // Every converged trial merged its words before it counted itself
            // done, so each word now holds the winner's (smallest key's) word.
            uint32_t *out = job.corr + row * job.corr_stride;
            const unsigned long long *src = sd.rec.win + rs * Wn;
            for (int w = 0; w < Wn; ++w) out[w] = (uint32_t)(__ldcg(src + w) & 0xffffffffull);
            job.conv[row] = 1;
            job.iters[row] = (int16_t)(best & 0xffffull);
            if (job.stage) job.stage[row] = 1;
        }
        // The record is free for a later failure once its reads are done.  Its claim
        // word is the next one's from here on (failure numbers go round the ring).
        const unsigned long long seq = ld_vol_u64(sd.rec.qseq + rs);
        if (!COLS && (sd.flags & kServe))
            atomicExch(sd.rec.claim + rs, claim_word(seq - 1ull + (unsigned long long)sd.rec.cap, 0));
        __threadfence();
        st_release_u64(sd.rec.qseq + rs, seq | kRecFree);
        shot_complete(sd, row, shot);
    }
}

// Under the first-success rule (select = 1) the winner is the earliest
// converged trial: once trial k* has converged, no later trial can win.
__device__ __forceinline__ bool trial_cannot_win(const StreamDev &sd, long long rs, int kidx) {
    if (sd.code.select != 1) return false;
    const unsigned long long best = __ldcg(sd.rec.best + rs);
    return best != ~0ull && (long long)(best >> 32) < (long long)kidx;
}

// Lane-parallel write-out of outboxes that need no warp cooperation:
// converged or uncorrectable initial runs, and trial runs.  (LONG: a converged
// initial run's words are out already.)
template <bool DEBUG, bool LONG, bool COLS>
__device__ __forceinline__ void finalize_simple(const StreamDev &sd, TeamMem T, int s, MgrState &mg) {
    const CodeDev &cd = sd.code;
    const JobDev &job = sd.job;
    const OutBox *ss = &T.ob[s];
    const int kind = ss->kind, iter = ss->iter;
    const bool conv = ss->outcome == 1;
    const long long shot = ss->shot;
    const long long row = row_of(sd, shot);
    const int Wn = cd.Wn;
    if (kind == 1) {
        mg.init_local += 1;
        // A failed run with trials already has its record and provisional
        // output (written by its team before it published the trials).
        if (!conv && cd.w > 0) return;
        uint32_t *out = job.corr + row * job.corr_stride;
        if (!LONG || !conv)
            for (int w = 0; w < Wn; ++w) out[w] = slot_word(T.ebits, Wn, s, w);
        job.conv[row] = conv ? 1 : 0;
        job.iters[row] = (int16_t)(conv ? iter : cd.max_iter);
        if (job.stage) job.stage[row] = conv ? 0 : 2;
        shot_complete(sd, row, shot);
        return;
    }
    // Trial run: undo the flip (Algorithm 1) and take part in the selection.
    const int C = cd.n_trials, kidx = ss->kidx;
    const long long rs = ss->rec;
    if (conv) {
        // e' xor t, in the slot's packed decision (the outbox is this lane's
        // until it is released): t flips the record's Phi[j] for the bits j
        // of the trial's mask.
        uint32_t *ew = T.ebits + s * Wn;
        const unsigned long long mask = __ldg(cd.trial_mask + kidx);
        for (int j0 = 0; j0 < cd.w; j0 += 8) {
            int b[8];
#pragma unroll
            for (int j = 0; j < 8; ++j)
                b[j] = j0 + j < cd.w && ((mask >> (j0 + j)) & 1ull) ? __ldcg(sd.rec.phi + rs * cd.w + j0 + j) : -1;
#pragma unroll
            for (int j = 0; j < 8; ++j)
                if (b[j] >= 0) ew[b[j] >> 5] ^= 1u << (b[j] & 31);
        }
        unsigned wsum = 0;
        for (int w = 0; w < Wn; ++w) wsum += __popc(ew[w]);
        // Selection key (unique per trial): weight, then list index; or the
        // list index alone under the first-success rule.
        const unsigned long long key = cd.select == 0 ? (((unsigned long long)wsum << 12) | (unsigned)kidx)
                                                      : (unsigned long long)kidx;
        const unsigned long long old = atomicMin(&sd.rec.best[rs], (key << 32) | (unsigned)iter);
        // Only a trial that held the smallest key so far merges its words: the
        // final winner always does, and merges of others cannot beat it.
        if ((old >> 32) > key) {
            unsigned long long *win = sd.rec.win + rs * Wn;
            for (int w = 0; w < Wn; ++w) atomicMin(win + w, (key << 32) | ew[w]);
        }
    }
    if (DEBUG) {
        if (sd.dbg.trial_conv) sd.dbg.trial_conv[shot * C + kidx] = conv ? 1 : 0;
        if (sd.dbg.trial_iters) sd.dbg.trial_iters[shot * C + kidx] = (int16_t)iter;
    }
    if (ss->outcome == 3)
        mg.trials_cancelled += 1;  // stopped: it could not win
    else
        mg.trials_local += 1;
    trial_done<COLS>(sd, rs, row, shot, conv);
}

// Shots that may be claimed now.
__device__ __forceinline__ long long shots_available(const StreamDev &sd) {
    if (sd.flags & kServe) return ld_acquire_sys_s64(sd.serve.published);
    return sd.job.n_shots;
}

// Fill the ready queue: trials first, then new shots.
//
// Trials are claimed from the records themselves: a record counts the trials
// taken from it (Records::done), and rec_head is the first failure whose record
// may have some left.  The lanes look at the 32 records from there on, the
// block picks among those with trials left by its number, and each record
// picked takes one addition, which always succeeds or shows the record used
// up.  (A server's records are reused: there it is a compare-and-swap, see
// claim_word.)  One ticket number for all, taken by compare and swap, failed for
// most of the blocks that raced for a failed shot's trials: 30 000 [[144]] shots
// at p = 0.05 took 2.4 ms, and 1.85 ms with this.
//
// While there are fewer trials than the launch has slots (128 when serving,
// where they go before new shots), a block takes no more of them than its idle
// slots, and while less than two launches full of shots are left, no more of
// these than its idle slots and about two shares of what is left.  The end of a
// batch, or all of a small one, so spreads over the blocks: 300 [[144]] shots
// at p = 0.05 took 0.37 ms with claims of up to 32 shots and take 0.34 ms;
// four failed [[254]] shots took 525 us with claims of up to 32 trials (two
// blocks then ran all 52) and take 102 us.
template <bool DEBUG, bool COLS>
__device__ __forceinline__ bool prefetch(const StreamDev &sd, unsigned char *qbase, int Q, int qstride, int lane,
                                         MgrState &mg, int n_empty, int nslots, unsigned long long head,
                                         unsigned long long rc, long long shot_next, unsigned long long wait_ns) {
    const CodeDev &cd = sd.code;
    const int Ws = cd.Ws;
    const bool serve = !COLS && (sd.flags & kServe);  // the column path never serves
    bool got_any = false;
    int space = Q - (mg.tail - mg.head);
    unsigned long long stall = 0ull;
    if (space > 0 && cd.w > 0 && !(sd.flags & kNoTickets)) {
        const int T = cd.n_trials;
        int lim = space < 32 ? space : 32;
        const unsigned long long few = serve ? 128ull : (unsigned long long)gridDim.x * (unsigned)nslots;
        if (rc < head + 1ull + few / (unsigned)T && lim > n_empty) lim = n_empty;
        if (head < rc && lim > 0) {
            const unsigned long long q = head + (unsigned long long)lane;
            long long rs = (long long)(q & (unsigned long long)(sd.rec.cap - 1));
            // The record holds failure q: q + 1; it did, and all its trials are done:
            // with the kRecFree bit; it holds a later one: above; else q is not written yet.
            const unsigned long long seq = q < rc ? ld_acquire_u64(sd.rec.qseq + rs) : 0ull;
            unsigned long long word = 0ull;
            int taken = T;
            if (seq == q + 1ull) {
                if (serve) word = ld_vol_u64(sd.rec.claim + rs);
                taken = serve ? claim_taken(word, q, T) : (int)(ld_vol_u32(sd.rec.done + rs) >> kDoneBits);
            }
            const bool left = taken < T;
            const bool unwritten = (seq & ~kRecFree) < q + 1ull;
            const unsigned lm = __ballot_sync(FULLMASK, left);
            // Records used up from the head on.
            const unsigned pm = __ballot_sync(FULLMASK, left || unwritten);
            const int used = pm ? __ffs(pm) - 1 : 32;
            if (lane == 0 && used > 0) atomicMax(&sd.ctr->rec_head, head + (unsigned long long)used);
            int k0 = 0, got = 0;  // first trial and number of trials taken from the lane's record
            if (lm) {
                const int n = __popc(lm), rank = __popc(lm & ((1u << lane) - 1u));
                int nth = rank - (int)(blockIdx.x % (unsigned)n);  // the lane's place in the block's order
                if (nth < 0) nth += n;
                const int want = lim - nth * T < T ? lim - nth * T : T;
                if (left && want > 0 && serve) {
                    got = claim_trials(word, q, want, T, &k0, [&](unsigned long long old, unsigned long long next) {
                        return atomicCAS(sd.rec.claim + rs, old, next);
                    });
                } else if (left && want > 0) {
                    k0 = (int)(atomicAdd(&sd.rec.done[rs], (unsigned)want << kDoneBits) >> kDoneBits);
                    got = T - k0 < want ? (T - k0 > 0 ? T - k0 : 0) : want;
                }
            }
            // Lane i takes the i-th trial: its record and number.
            int before = got;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(FULLMASK, before, o);
                if (lane >= o) before += y;
            }
            const int take = __shfl_sync(FULLMASK, before, 31);
            before -= got;
            int kidx = 0;
            long long mine_rs = 0;
            for (unsigned m = __ballot_sync(FULLMASK, got > 0); m; m &= m - 1u) {
                const int s = __ffs(m) - 1;
                const int b = __shfl_sync(FULLMASK, before, s), g = __shfl_sync(FULLMASK, got, s);
                const int k = __shfl_sync(FULLMASK, k0, s);
                const long long r = __shfl_sync(FULLMASK, rs, s);
                if (lane >= b && lane < b + g) {
                    kidx = k + lane - b;
                    mine_rs = r;
                }
            }
            __syncwarp();  // the claiming lane's acquire of the record holds for the lanes that read it
            if (lane < take) {
                rs = mine_rs;
                QEntry *e = qentry(qbase, (mg.tail + lane) % Q, qstride);
                const long long shot = __ldcg(sd.rec.qshot + rs);
                if (!trial_cannot_win(sd, rs, kidx)) {
                    e->kind = 2;
                    e->kidx = (int16_t)kidx;
                    e->rec = (int)rs;
                    e->shot = shot;
                    // The trial vector t: the bits Phi[j] its mask selects.
                    const unsigned long long mask = __ldg(cd.trial_mask + kidx);
                    uint32_t *sy = qsyn(e);
                    for (int w = 0; w < Ws; ++w) sy[w] = __ldcg(sd.rec.synd + rs * Ws + w);
                    // s' = s xor t H^T (Algorithm 1): flip the checks of every
                    // selected bit (eight entries of Phi are loaded at a time).
                    for (int j0 = 0; j0 < cd.w; j0 += 8) {
                        int v[8];
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            v[j] = j0 + j < cd.w && ((mask >> (j0 + j)) & 1ull) ? __ldcg(sd.rec.phi + rs * cd.w + j0 + j) : -1;
#pragma unroll
                        for (int j = 0; j < 8; ++j) {
                            if (v[j] < 0) continue;
                            for (int k = 0; k < cd.vstride; ++k) {
                                const int c = __ldg(cd.vchk + v[j] * cd.vstride + k);
                                if (c == 0xffff) break;
                                sy[c >> 5] ^= 1u << (c & 31);
                            }
                        }
                    }
                    if (DEBUG && sd.dbg.trial_synd)
                        for (int w = 0; w < Ws; ++w) sd.dbg.trial_synd[(shot * T + kidx) * Ws + w] = sy[w];
                } else {
                    // Early cancel: counted as done, not run.
                    trial_done<COLS>(sd, rs, row_of(sd, shot), shot, false);
                    ++mg.trials_cancelled;
                    e->kind = 0;
                }
            }
            __syncwarp();
            mg.tail += take;
            space -= take;
            got_any = take > 0;
            // The first record is announced but not written yet: looked at again in
            // the next pass, and given up and reported when that lasts too long.
            if (used == 0 && !(lm & 1u)) {
                const unsigned long long now = globaltimer_ns();
                stall = head + 1ull;
                if (mg.stall_q != stall) mg.stall_since = now;
                if (now - mg.stall_since > wait_ns) {
                    if (lane == 0) {
                        atomicOr(&sd.ctr->status, kDevReadyTimeout);
                        atomicMax(&sd.ctr->rec_head, head + 1ull);
                    }
                    stall = 0ull;
                }
            }
        }
    }
    mg.stall_q = stall;
    if (space > 0 && (serve || shot_next < sd.job.n_shots)) {
        long long c0 = 0;
        int got = 0;
        if (lane == 0) {
            const long long avail = shots_available(sd);
            long long cur = shot_next;
            for (int att = 0; att < 4 && cur < avail; ++att) {
                const long long left = avail - cur, grid = (long long)gridDim.x;
                long long want = space < 32 ? space : 32;
                if (left < 2 * grid * nslots) {
                    const long long share = 1 + 2 * left / grid;
                    want = want < share ? want : share;
                    want = want < n_empty ? want : n_empty;
                    if (want == 0) break;
                }
                if (serve) {
                    // More shots may be published later: claim none that are not yet.
                    if (want > left) want = left;
                    const long long seen = (long long)atomicCAS(&sd.ctr->shot_next, (unsigned long long)cur,
                                                                (unsigned long long)(cur + want));
                    if (seen != cur) {
                        cur = seen;
                        continue;
                    }
                    c0 = cur;
                    got = (int)want;
                } else {
                    c0 = (long long)atomicAdd(&sd.ctr->shot_next, (unsigned long long)want);
                    const long long hi = (c0 + want) < avail ? (c0 + want) : avail;
                    got = c0 < avail ? (int)(hi - c0) : 0;
                }
                break;
            }
        }
        c0 = __shfl_sync(FULLMASK, c0, 0);
        got = __shfl_sync(FULLMASK, got, 0);
        // Lane 0's acquire of the published count orders the other lanes'
        // reads of the rows too (when serving, the host writes the rows
        // before it publishes them).
        __syncwarp();
        if (lane < got) {
            const long long shot = c0 + lane;
            QEntry *e = qentry(qbase, (mg.tail + lane) % Q, qstride);
            e->kind = 1;
            e->kidx = 0;
            e->rec = -1;
            e->shot = shot;
        }
        // The syndromes' words, spread over the lanes; four loads of a lane are under way at a time.
        const int words = got * Ws;
        for (int k0 = lane; k0 < words; k0 += 128) {
            uint32_t v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + 32 * u, sh = k / Ws;
                if (k < words) v[u] = __ldcg(sd.job.synd + row_of(sd, c0 + sh) * sd.job.synd_stride + (k - sh * Ws));
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = k0 + 32 * u, sh = k / Ws;
                if (k < words) qsyn(qentry(qbase, (mg.tail + sh) % Q, qstride))[k - sh * Ws] = v[u];
            }
        }
        __syncwarp();
        mg.tail += got;
        got_any = got_any || got > 0;
    }
    return got_any;
}

template <bool DEBUG, bool LONG, bool COLS>
__device__ void manager_loop(const StreamDev &sd, const LayoutMem &L, unsigned char *team_base, int team_bytes,
                             const TeamOffsets &to, int teams, int S, unsigned char *qbase, int Q, BlockHdr *hdr,
                             int lane, unsigned long long wait_ns) {
    const CodeDev &cd = sd.code;
    const int qstride = qentry_bytes(cd.Ws);
    const int nslots = teams * S, lgS = __ffs(S) - 1;
    const bool serve = (sd.flags & kServe) != 0;
    MgrState mg{0, 0, 0u, 0u, 0u, 0ull, 0ull};
    unsigned idle_ns = 32;     // back-off after passes that found nothing to do
    unsigned idle_passes = 0;  // consecutive passes without progress
    for (;;) {
        bool progress = false;
        bool busy = false;
        int n_empty = 0;  // idle slots of the block with an empty inbox (warp-uniform)
        if (lane == 0) hdr->heartbeat = hdr->heartbeat + 1u;
        // (A) write out the outboxes the teams filled.
        for (int g0 = 0; g0 < nslots; g0 += 32) {
            const int g = g0 + lane;
            const bool inr = g < nslots;
            const int t = inr ? g >> lgS : 0, s = g & (S - 1);
            TeamMem T = team_mem(team_base + t * team_bytes, to);
            const int stv = inr ? *vstate(&T.st[s]) : kSlotEmpty;
            const bool fin = inr && *vflag(&T.ob[s].full) != 0;
            __threadfence_block();
            if (__any_sync(FULLMASK, stv != kSlotEmpty)) busy = true;
            // First-success rule: ask running trials that can no longer win to stop.
            if (cd.select == 1 && stv == kSlotRunning && T.st[s].kind == 2) {
                const long long shot = T.st[s].shot;
                const int kidx = T.st[s].kidx;
                const long long key = shot * (long long)cd.n_trials + kidx + 1;
                if (T.st[s].cancel != key && trial_cannot_win(sd, T.st[s].rec, kidx))
                    *reinterpret_cast<volatile long long *>(&T.st[s].cancel) = key;
            }
            if (fin) finalize_simple<DEBUG, LONG, COLS>(sd, T, s, mg);
            __syncwarp();
            if (fin) {
                __threadfence_block();
                *vflag(&T.ob[s].full) = 0;
            }
            if (__any_sync(FULLMASK, fin)) progress = true;
        }
        __syncwarp();
        // The counters that (C) needs, on their way while (B) runs.
        const unsigned long long rec_head = ld_vol_u64(&sd.ctr->rec_head), rec_count = ld_vol_u64(&sd.ctr->rec_count);
        const long long shot_next = (long long)ld_vol_u64(&sd.ctr->shot_next);
        // (B) fill empty inboxes from the ready queue: idle slots first (they
        // start at once), then running ones (their next run).  Count the
        // slots left idle with nothing in their inbox.
        for (int pass = 0; pass < 2; ++pass) {
            for (int g0 = 0; g0 < nslots && (pass == 1 || mg.tail > mg.head); g0 += 32) {
                const int g = g0 + lane;
                const bool inr = g < nslots;
                const int t = inr ? g >> lgS : 0, s = g & (S - 1);
                TeamMem T = team_mem(team_base + t * team_bytes, to);
                const bool idle = inr && *vstate(&T.st[s]) == kSlotEmpty;
                const bool open = inr && *vflag(&T.ibf[s]) == 0 && (pass == 1 || idle);
                const unsigned om = __ballot_sync(FULLMASK, open);
                const int rank = __popc(om & ((1u << lane) - 1u));
                const int avail = mg.tail - mg.head;
                const bool take = open && rank < avail;
                if (take) {
                    const uint4 *src = reinterpret_cast<const uint4 *>(qentry(qbase, (mg.head + rank) % Q, qstride));
                    uint4 *dst = reinterpret_cast<uint4 *>(T.ib + s * T.ibstride);
                    for (int k = 0; k < qstride / 16; ++k) dst[k] = src[k];
                    __threadfence_block();
                    *vflag(&T.ibf[s]) = 1;
                }
                const int used = __popc(om) < avail ? __popc(om) : avail;
                mg.head += used;
                if (used) progress = true;
                if (pass == 1) n_empty += __popc(__ballot_sync(FULLMASK, open && !take && idle));
            }
        }
        __syncwarp();
        // (C) claim work ahead.
        if (prefetch<DEBUG, COLS>(sd, qbase, Q, qstride, lane, mg, n_empty, nslots, rec_head, rec_count, shot_next, wait_ns))
            progress = true;
        // Count finished initial runs once no new shot can be claimed.
        if (!serve && shot_next >= sd.job.n_shots) {
            const unsigned tot = __reduce_add_sync(FULLMASK, mg.init_local);
            mg.init_local = 0;
            if (lane == 0 && tot) {
                __threadfence();
                atomicAdd(&sd.ctr->init_done, (unsigned long long)tot);
            }
        }
        // (D) leave when nothing is running, queued, boxed or claimable.
        if (!busy && !progress && mg.stall_q == 0ull && mg.tail == mg.head) {
            bool any_slot = false;
            for (int g0 = 0; g0 < nslots; g0 += 32) {
                const int g = g0 + lane;
                const int t = g < nslots ? g >> lgS : 0, s = g & (S - 1);
                TeamMem T = team_mem(team_base + t * team_bytes, to);
                // Read order matters: inbox flag, state, outbox flag (the
                // team writes state before clearing the inbox flag, and the
                // outbox flag before the state).
                bool occ = false;
                if (g < nslots) {
                    occ = *vflag(&T.ibf[s]) != 0;
                    __threadfence_block();
                    occ = occ || *vstate(&T.st[s]) != kSlotEmpty;
                    __threadfence_block();
                    occ = occ || *vflag(&T.ob[s].full) != 0;
                }
                if (__any_sync(FULLMASK, occ)) any_slot = true;
            }
            // Nothing left for this code: hand the block back, which then
            // waits across all codes (serving) or for other blocks' trials.
            if (!any_slot) break;
        }
        // A run of passes that find nothing backs off, up to 1 us (a finished
        // slot then waits that long at most for its write-out); any progress
        // resets it.
        if (progress) {
            idle_ns = 32;
            idle_passes = 0;
        } else {
            __nanosleep(idle_ns);
            if (++idle_passes > kIdleLooks) idle_ns = idle_ns < 1024 ? 2 * idle_ns : 1024;
        }
    }
    // Flush counters and release the teams.
    const unsigned init_tot = __reduce_add_sync(FULLMASK, mg.init_local);
    const unsigned trial_tot = __reduce_add_sync(FULLMASK, mg.trials_local);
    const unsigned skip_tot = __reduce_add_sync(FULLMASK, mg.trials_cancelled);
    if (lane == 0) {
        if (init_tot) {
            __threadfence();
            atomicAdd(&sd.ctr->init_done, (unsigned long long)init_tot);
        }
        if (trial_tot) atomicAdd(&sd.ctr->trial_runs, (unsigned long long)trial_tot);
        if (skip_tot) atomicAdd(&sd.ctr->trials_cancelled, (unsigned long long)skip_tot);
        unsigned long long it = 0, cap = 0;
        for (int t = 0; t < teams; ++t) {
            TeamMem T = team_mem(team_base + t * team_bytes, to);
            it += T.ctl->iters;
            cap += T.ctl->cap;
            T.ctl->iters = 0;
            T.ctl->cap = 0;
        }
        if (it) atomicAdd(&sd.ctr->iters_total, it);
        if (cap) atomicAdd(&sd.ctr->slot_capacity, cap);
        __threadfence_block();
        hdr->exit = 1;
    }
    __syncwarp();
}

// MINB: minimum resident blocks per SM the register allocation must allow.
// Two caps registers at 64 per thread, so two 512-thread blocks (or three
// smaller ones) fit on an SM; one keeps the full budget, which four slots
// per lane need.  The exact-degree variant has both instances (the launch
// plan picks by the blocks that fit); the others (wider rows, irregular
// codes whose shared-memory needs allow few slots per SM anyway) have one.
#ifndef BPSF_MIN_BLOCKS
#define BPSF_MIN_BLOCKS 2
#endif

// LAY: the instance also runs codes with the layered schedule (a launch
// with no such code uses the instance without that path and its registers).
// FB: bytes per flip word (FlipW): 2, or 1 for launches whose codes all have
// max_iter <= 127 (an instance that leaves more shared memory for slots).
// MIX: the instance also carries the exact (6, 4, 3) team loop and runs it
// for codes with exactly six ones per row and three per column, so such codes
// keep their specialised path in a launch that mixes them with codes of
// wider rows (the layouts agree: both have column tables of width DVS).
template <int DC, int DVS, int DVX, bool DEBUG, int MINB, bool LAY, int FB = 2, bool MIX = false, bool COLS = false>
__global__ void __launch_bounds__(COLS ? (DVX > 0 ? kColumnThreads : kLongThreads) : 512, MINB) bpsf_persistent(const __grid_constant__ KernelParams kp) {
    constexpr int kPath = !COLS ? kPathTeams : (DVX > 0 ? kPathColumns : kPathLong);
    extern __shared__ __align__(16) unsigned char smem[];
    BlockHdr *hdr = reinterpret_cast<BlockHdr *>(smem);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int Q = kp.Q;
    int cur = -1;
    bool waiting = false;
    unsigned long long wait_start = 0;
    for (;;) {
        if (warp == 0) {
            // Lane k looks at stream k, so the streams' counters are read in one
            // round trip.  A block stays with its stream while there is work to
            // claim there; when it has to move, the blocks spread over the streams
            // that still have work (block b takes the (b mod n)-th of the n).
            // Taking the next one in order instead sent the blocks of a finished
            // job to one shard of the next job, whose counters they then queued on:
            // four [[144]] jobs (p = 0.02 .. 0.08, 250 000 shots each) in one launch
            // took 135.6 ms that way, and the four one after another 101 ms.
            bool claimable = false, done = true;
            if (lane < kp.n_streams) {
                const StreamDev &sd = kp.streams[lane];
                const StreamCounters *c = sd.ctr;
                if (sd.flags & kServe) {
                    const long long pub = ld_acquire_sys_s64(sd.serve.published);
                    const long long sn = (long long)ld_vol_u64(&c->shot_next);
                    claimable = sn < pub || ld_vol_u64(&c->rec_head) < ld_vol_u64(&c->rec_count);
                    done = !claimable && *sd.serve.stop;
                } else {
                    const unsigned long long n = (unsigned long long)sd.job.n_shots;
                    const unsigned long long shot_next = ld_vol_u64(&c->shot_next);
                    const unsigned long long init_done = ld_vol_u64(&c->init_done);
                    __threadfence();
                    const unsigned long long rc = ld_vol_u64(&c->rec_count);
                    const unsigned long long rh = ld_vol_u64(&c->rec_head);
                    const bool trials = sd.code.w > 0 && !(sd.flags & kNoTickets);
                    const bool left = trials && rh < rc;
                    claimable = shot_next < n || left;
                    done = shot_next >= n && init_done >= n && !left;
                }
            }
            const unsigned cm = __ballot_sync(FULLMASK, claimable);
            const bool all_done = __all_sync(FULLMASK, done);
            if (lane == 0) {
                int pick = -1;
                if (cur >= 0 && ((cm >> cur) & 1u)) {
                    pick = cur;
                } else if (cm) {
                    pick = (int)__fns(cm, 0u, (int)(blockIdx.x % (unsigned)__popc(cm)) + 1);
                }
                hdr->stream = pick;
                hdr->cmd = pick >= 0 ? 1 : (all_done ? 2 : 0);
            }
        }
        __syncthreads();
        const int cmd = hdr->cmd, sid = hdr->stream;
        __syncthreads();
        if (cmd == 2) break;
        if (cmd == 0) {
            // Other blocks still run initial runs that may publish trials, or
            // a serving loop waits for requests.
            if (tid == 0) {
                const unsigned long long now = globaltimer_ns();
                bool serve_any = false, serve_quit = true;
                for (int k = 0; k < kp.n_streams; ++k)
                    if (kp.streams[k].flags & kServe) {
                        serve_any = true;
                        if (!*kp.streams[k].serve.stop &&
                            (!waiting || now - wait_start <= (unsigned long long)kp.streams[k].serve.idle_ns))
                            serve_quit = false;
                    }
                if (!waiting) {
                    waiting = true;
                    wait_start = now;
                } else if (serve_any) {
                    if (serve_quit) hdr->cmd = 3;
                } else if (now - wait_start > kp.wait_ns) {
                    for (int k = 0; k < kp.n_streams; ++k) atomicOr(&kp.streams[k].ctr->status, kDevIdleTimeout);
                    hdr->cmd = 3;
                }
                __nanosleep(1000);
            }
            __syncthreads();
            const int quit = hdr->cmd == 3;
            __syncthreads();
            if (quit) break;
            continue;
        }
        waiting = false;
        if (COLS && sid != cur) {
            // The column path reads its descriptor in shared memory.
            const uint32_t *src = reinterpret_cast<const uint32_t *>(&kp.streams[sid]);
            for (int k = tid; k < (int)(sizeof(StreamDev) / 4); k += blockDim.x)
                reinterpret_cast<uint32_t *>(smem + kBlockHeaderBytes)[k] = src[k];
            const StreamDev &d = kp.streams[sid];
            if (tid == 0)
                *reinterpret_cast<TeamOffsets *>(smem + kBlockHeaderBytes + kStreamBytes) =
                    team_offsets(d.S, d.code.M, d.code.N, d.code.P, d.code.Ws, 0, FB, kPath);
            __syncthreads();
        }
        const StreamDev &sd = COLS ? *reinterpret_cast<const StreamDev *>(smem + kBlockHeaderBytes) : kp.streams[sid];
        const CodeDev &cd = sd.code;
        const int S = sd.S, W = sd.W, teams = sd.teams;
        const LayoutOffsets lo = layout_offsets(cd.M, cd.N, DVS, cd.P, kPath);
        unsigned char *lay = smem + kBlockHeaderBytes + (COLS ? kDescriptorBytes : 0);
        if (sid != cur && kPath != kPathColumns) {
            uint8_t *rd = lay + lo.row_deg;
            uint16_t *vp = reinterpret_cast<uint16_t *>(lay + lo.vpos);
            float *lc = reinterpret_cast<float *>(lay + lo.lch);
            float *lp = reinterpret_cast<float *>(lay + lo.lch_pos);
            for (int k = tid; k < cd.M; k += blockDim.x) rd[k] = cd.row_deg[k];
            for (int k = tid; k < cd.N * DVS; k += blockDim.x) vp[k] = cd.vpos[k];
            for (int k = tid; k < cd.N; k += blockDim.x) lc[k] = cd.lch[k];
            for (int k = tid; kPath == kPathTeams && k < cd.P; k += blockDim.x) lp[k] = cd.lch_pos[k];
        }
        const bool fill = sid != cur;
        cur = sid;
        // Every slot starts empty; teams start idle.
        TeamOffsets to_reg;
        if (!COLS) to_reg = team_offsets(S, cd.M, cd.N, cd.P, cd.Ws, cd.layered, FB);
        const TeamOffsets &to =
            COLS ? *reinterpret_cast<const TeamOffsets *>(smem + kBlockHeaderBytes + kStreamBytes) : to_reg;
        unsigned char *qbase = lay + lo.total;
        unsigned char *team_base = qbase + Q * qentry_bytes(cd.Ws);
        for (int k = tid; k < teams * S; k += blockDim.x) {
            unsigned char *tb = team_base + (k / S) * to.total;
            SlotState *ss = reinterpret_cast<SlotState *>(tb + to.state) + (k % S);
            ss->state = kSlotEmpty;
            ss->kind = 0;
            ss->cancel = 0;
            reinterpret_cast<OutBox *>(tb + to.outbox)[k % S].full = 0;
            reinterpret_cast<int *>(tb + to.inflag)[k % S] = 0;
        }
        for (int t = tid; t < teams; t += blockDim.x) {
            TeamCtl *ctl = reinterpret_cast<TeamCtl *>(team_base + t * to.total + to.ctl);
            ctl->iters = 0;
            ctl->cap = 0;
            ctl->exit = 0;
        }
        // Syndrome and residual-syndrome words start at zero: installs toggle
        // only their own slot's bits, and the padding bits past S*M are read
        // by the convergence test.
        {
            const int sw = (to.ebits - to.syn) / 4;
            for (int k = tid; k < teams * sw; k += blockDim.x) {
                const int t = k / sw, w = k - t * sw;
                reinterpret_cast<uint32_t *>(team_base + t * to.total + to.syn)[w] = 0u;
            }
        }
        // Messages that no install sets up (uniform channel LLRs) start finite: the
        // first iteration multiplies them by zero.
        if (kPath == kPathTeams && cd.uniform && !cd.layered && fill) {
            const int words = to.m + 4 * S * cd.P;
            for (int t = 0; t < teams; ++t)
                for (int k = to.m / 4 + tid; k < words / 4; k += blockDim.x)
                    reinterpret_cast<uint32_t *>(team_base + t * to.total)[k] = 0u;
        }
        if (tid == 0) {
            hdr->exit = 0;
            hdr->heartbeat = 0u;
            hdr->wait_ns = kp.wait_ns;
        }
        __syncthreads();
        LayoutMem L;
        L.row_deg = lay + lo.row_deg;
        L.vpos = reinterpret_cast<const uint16_t *>(lay + lo.vpos);
        L.lch = reinterpret_cast<const float *>(lay + lo.lch);
        L.lch_pos = reinterpret_cast<const float *>(lay + lo.lch_pos);
        if (warp == 0) {
            manager_loop<DEBUG, kPath == kPathLong, COLS>(sd, L, team_base, to.total, to, teams, S, qbase, Q, hdr, lane, kp.wait_ns);
        } else {
            const int team = (warp - 1) / W;
            if (team < teams) {
                TeamMem T = team_mem(team_base + team * to.total, to);
                const int ttid = tid - 32 - team * W * 32;
                if constexpr (COLS) {
                    const int tb = keep((int)(team_base - smem) + team * to.total);
                    if constexpr (DVX == 0)
                        column_loop<DC, 3, DVS, kLongSlots, true, DEBUG, FB>(sd, to, hdr, L, tb, W, ttid, 1 + team);
                    else if (S == 4)
                        column_loop<DC, DVX, DVS, 4, false, DEBUG, FB>(sd, to, hdr, L, tb, W, ttid, 1 + team);
                    else
                        column_loop<DC, DVX, DVS, 1, false, DEBUG, FB>(sd, to, hdr, L, tb, W, ttid, 1 + team);
                } else if (MIX && cd.regular && cd.DC == 6 && cd.dv_max == 3)
                    team_loop<6, DVS, 3, DEBUG, MINB, LAY, FB>(sd, L, T, hdr, S, W, ttid, 1 + team, kp.wait_ns);
                else
                    team_loop<DC, DVS, DVX, DEBUG, MINB, LAY, FB>(sd, L, T, hdr, S, W, ttid, 1 + team, kp.wait_ns);
            }
        }
        __syncthreads();
    }
}

}  // namespace bpsf
