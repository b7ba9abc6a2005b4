// Persistent coupled photon-electron transport kernel for sm_103a.
//
// One launch runs every particle it can reach to completion.  Each warp holds
// 32 particles of ONE type (photon or electron) in registers and advances all
// of them together: up to four Woodcock flights and the real event they end on
// for photons (GPUMCD §II.A), up to four condensed-history steps for electrons
// (§II.B.3).  Lanes whose
// particle ended are refilled, in this order, from the warp's private stack of
// that type, from the global overflow queue of the previous launch, and from
// the primaries of the launch's plans (claimed in chunks).  Secondaries go to
// the warp's private stacks (the paper's per-type particle arrays, §II.C.2)
// and spill to a global overflow queue only when a stack fills; a warp
// switches type when its own lanes run dry or when the other stack is high
// (§II.C.3's "pool" of persistent threads, with warp-uniform particle type).
// An electron step that ends on a hard-event candidate parks the particle on
// a third per-warp stack; with 32 parked, the warp runs their Woodcock tests
// and Moller/bremsstrahlung events together (a converged hard pass) instead
// of one or two lanes at a time inside every step.
//
// Randomness is a counter-based Philox keyed by the plan seed with counter
// (draw, lineage lo, lineage hi, history), and energies are integers, so the
// tally is independent of how particles are scheduled.
//
// Divisions on the event path are written __fdividef (reciprocal, then
// multiply): every divisor there is a direction cosine, an energy, a cross
// section or a sampler constant, far inside the range (|y| < 2^126) for which
// that form is specified.  There it skips the range handling of the
// approximate division this file is compiled with (-prec-div=false), and the
// tallies and event counts of every workload compared were bit-identical with
// either form.
#include "gm_common.cuh"
#include "gm_host.h"

namespace gm {

// Relative margin of the per-voxel electron hard-event majorant (2^-14).
constexpr float kHardMajorantMargin = 1.00006103515625f;
constexpr unsigned FULL = 0xffffffffu;
constexpr int MAX_WARPS = 32;
// A warp's row of event counters: those before the cycle profile, then the hard passes.
constexpr int CNT_ROW = CNT_PROF_CYC + 1;
__host__ __device__ constexpr int row_word(int which) { return which == CNT_HARD_PASSES ? CNT_ROW - 1 : which; }

struct WarpState {
    unsigned int stk[2];
    unsigned int hc;   // parked hard-event candidates (electrons)
    unsigned int pad;
    unsigned long long p_lo[2], p_hi[2];  // claimed primaries by type (type-local index)
    unsigned long long q_lo[2], q_hi[2];  // claimed overflow-queue records by type
};

struct Lane {
    float x, y, z, ux, uy, uz;
    uint32_t E, hist, draw, plan;
    PhiloxLineage lin;
    bool act;
};

// Shared-memory context of a CTA.
struct Smem {
    const float *tab;
    PlanDev *plans;
    WarpState *ws;
    unsigned int *wcnt;          // [MAX_WARPS][CNT_ROW] event counters, a row per warp
    unsigned long long *cnt;     // [CNT_N] cycle profile (64-bit)
    unsigned int *ledger;        // [n_plans][3][2]: incident, escaped, rest; low and high words
};

__device__ __forceinline__ float interp(const float *t, float x) {
    x = fminf(fmaxf(x, 0.0f), (float)(G - 1));
    const int i = min((int)x, G - 2);
    const float f = x - (float)i;
    const float a = t[i], b = t[i + 1];
    return fmaf(f, b - a, a);
}

__device__ __forceinline__ float interp_ldg(const float *t, float x) {
    x = fminf(fmaxf(x, 0.0f), (float)(G - 1));
    const int i = min((int)x, G - 2);
    const float f = x - (float)i;
    const float a = __ldg(t + i), b = __ldg(t + i + 1);
    return fmaf(f, b - a, a);
}

__device__ __forceinline__ float interp_ms(const float *t, float x) {
    x = fminf(fmaxf(x, 0.0f), (float)(G_MS - 1));
    const int i = min((int)x, G_MS - 2);
    const float f = x - (float)i;
    return fmaf(f, t[i + 1] - t[i], t[i]);
}

// A plan's Philox round keys: computed from the plan's key (18 additions a
// draw), or, in a launch of one plan (ONE), operands of the rounds' exclusive
// ors in the kernel's arguments.  A draw's ten rounds are about a quarter of
// the transport's time (a build with six is 9-11% faster).  ONE takes 1e6 15
// MeV electrons on 128^3 water from 1.77 to 1.74 ms, 4e6 photons from 4.10 to
// 4.00 ms, 4e6 photons on the slabs from 3.12 to 3.05 ms, and spills less (4
// bytes a thread are loaded back instead of 12).
// Only the keys are read there: with the plan's other fields in the arguments
// too, the compiler contracts other multiply-adds (the tallies move) and the
// beams above take 0.4% more to 1.8% less than without ONE.
template <bool ONE>
struct RoundKeys {
    const TransportArgs &A;
    const PlanDev &P;
    __device__ __forceinline__ uint2 operator()(int r) const {
        return ONE ? A.round_key[r] : philox_round_key(make_uint2(P.key_lo, P.key_hi), r);
    }
};

template <class Keys>
__device__ __forceinline__ uint4 draw4(Lane &p, const Keys &key) {
    const uint4 r = philox4x32_10_lineage(p.draw, p.hist, p.lin, key);
    ++p.draw;
    return r;
}

// Lineage of the j-th particle a parent creates at draw index `draw`: a 64-bit
// finalizer of (parent lineage, draw, j), never equal to the primary's lineage 1.
template <class Keys>
__device__ __forceinline__ void child_lineage(const Lane &p, uint32_t j, const Keys &key, uint32_t &lo, uint32_t &hi) {
    const uint2 own = philox_lineage_words(p.lin.a, p.lin.c, key(0), key(1));
    unsigned long long z = ((unsigned long long)own.y << 32) | own.x;
    z ^= ((unsigned long long)p.draw << 20) ^ ((unsigned long long)(j + 1) << 52) ^ 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 33)) * 0xFF51AFD7ED558CCDull;
    z = (z ^ (z >> 33)) * 0xC4CEB9FE1A85EC53ull;
    z ^= z >> 33;
    z |= 2ull;
    lo = (uint32_t)z;
    hi = (uint32_t)(z >> 32);
}

__device__ __forceinline__ bool inside(const PlanDev &P, float x, float y, float z) {
    return x >= 0.f && y >= 0.f && z >= 0.f && x < P.X && y < P.Y && z < P.Z;
}

__device__ __forceinline__ uint32_t voxel_index(const PlanDev &P, float x, float y, float z, int &ix,
                                                int &iy, int &iz) {
    ix = min((int)(x * P.inv_dx), P.nx - 1);
    iy = min((int)(y * P.inv_dy), P.ny - 1);
    iz = min((int)(z * P.inv_dz), P.nz - 1);
    return (uint32_t)ix + (uint32_t)P.nx * ((uint32_t)iy + (uint32_t)P.ny * (uint32_t)iz);
}

// Distance along the direction to the exit face of voxel (ix, iy, iz).
__device__ __forceinline__ float exit_distance(const PlanDev &P, const Lane &p, int ix, int iy, int iz) {
    float dv = 3.0e38f;
    if (p.ux != 0.f) dv = fminf(dv, __fdividef(((p.ux > 0.f ? (float)(ix + 1) : (float)ix) - p.x * P.inv_dx) * P.dx, p.ux));
    if (p.uy != 0.f) dv = fminf(dv, __fdividef(((p.uy > 0.f ? (float)(iy + 1) : (float)iy) - p.y * P.inv_dy) * P.dy, p.uy));
    if (p.uz != 0.f) dv = fminf(dv, __fdividef(((p.uz > 0.f ? (float)(iz + 1) : (float)iz) - p.z * P.inv_dz) * P.dz, p.uz));
    return dv;
}

// One float further along a direction cosine.  An electron step ends a nudge
// past the face it aims at, but at a grazing angle nudge x cosine can fall
// below FP32 resolution and the end point rounds back onto the face; indexed
// by position, a particle crossing in the negative direction would then stay
// in the voxel it is leaving, with a zero distance to its exit, and creep on
// in nudge-sized steps (seen in thin air, where nothing deflects it).  Moving
// every end coordinate one float along its direction takes it off the face.
__device__ __forceinline__ float float_along(float x, float u) {
    const int b = __float_as_int(x);
    return u > 0.f ? __int_as_float(b + 1) : (u < 0.f ? __int_as_float(b - 1) : x);
}

// Fire-and-forget 64-bit add into the tally (no value comes back).
__device__ __forceinline__ void red_add_u64(unsigned long long *addr, unsigned long long v) {
    asm volatile("red.relaxed.gpu.global.add.u64 [%0], %1;" ::"l"(addr), "l"(v) : "memory");
}

__device__ __forceinline__ void deposit(const PlanDev &P, uint32_t hist, uint32_t idx, uint32_t e) {
    if (e == 0u) return;
    const uint32_t b = hist & P.bmask;  // batch = history mod W
    red_add_u64(P.tally + (size_t)b * P.nvox + idx, (unsigned long long)e);
}

// Deposit at a convergent point (all 32 lanes call it): lanes that hit the
// same tally word add their energies into one atomic.  Energies are < 2^31,
// so the group sum is formed exactly from two 32-bit reductions.
__device__ __forceinline__ void deposit_aggregated(const PlanDev &P, uint32_t hist, uint32_t idx,
                                                   uint32_t e) {
    const bool on = e != 0u;
    const unsigned mask = __ballot_sync(FULL, on);
    if (!on) return;
    const uint32_t b = hist & P.bmask;  // batch = history mod W
    unsigned long long *addr = P.tally + (size_t)b * P.nvox + idx;
    const unsigned peers = __match_any_sync(mask, (unsigned long long)addr);
    const unsigned lo = __reduce_add_sync(peers, e & 0xFFFFu);
    const unsigned hi = __reduce_add_sync(peers, e >> 16);
    if ((threadIdx.x & 31) == __ffs(peers) - 1)
        red_add_u64(addr, ((unsigned long long)hi << 16) + (unsigned long long)lo);
}

__device__ __forceinline__ void ledger_add(const Smem &S, uint32_t plan, int which, uint32_t e) {
    unsigned int *l = &S.ledger[(plan * 3 + which) * 2];
    if (atomicAdd(l, e) + e < e) atomicAdd(l + 1, 1u);  // the low word wrapped: carry
}

// A warp's event counter: at most 128 increments an iteration (EL_STEPS steps or
// PH_FLIGHTS flights of 32 lanes, or the records spilled) and at most 2^24 iterations a launch,
// so 32 bits hold it.  Counters and ledgers are 32-bit words because shared
// memory adds 32 bits in one instruction, without a result to wait for, while
// a 64-bit shared add is a compare-and-swap loop: its lanes retry one after
// another, and so did the 32 warps of the CTA on the counter they shared.
// With a row of counters per warp, and ledgers as a low word with a carry, the
// 15 MeV beams on 128^3 water take 2.11 ms (1e6 electrons) and 4.48 ms (4e6
// photons) of transport, 2.38 and 5.33 before; the 2 MeV pencil of 1e5
// photons 0.134 ms, 0.192 before.
__device__ __forceinline__ unsigned int *counter(const Smem &S, int w, int which) {
    return &S.wcnt[w * CNT_ROW + row_word(which)];
}
__device__ __forceinline__ void count(const Smem &S, int w, int which) { atomicAdd(counter(S, w, which), 1u); }

// Rotate (ux, uy, uz) by polar angle (cos c, sin s) and azimuth (cos cp, sin sp).
__device__ __forceinline__ void rotate(float &ux, float &uy, float &uz, float c, float s, float cp,
                                       float sp) {
    const float r2 = ux * ux + uy * uy;
    float nx, ny, nz;
    if (r2 > 1e-10f) {
        const float ir = rsqrtf(r2);
        const float r = r2 * ir;
        nx = ux * c + s * (ux * uz * cp - uy * sp) * ir;
        ny = uy * c + s * (uy * uz * cp + ux * sp) * ir;
        nz = uz * c - s * cp * r;
    } else {
        nx = s * cp;
        ny = s * sp;
        nz = uz >= 0.f ? c : -c;
    }
    const float n = rsqrtf(nx * nx + ny * ny + nz * nz);
    ux = nx * n;
    uy = ny * n;
    uz = nz * n;
}

// Push a new particle onto the warp's private stack of its type (headroom is
// guaranteed by the caller before each step).
template <bool ONE>
__device__ __forceinline__ void push(const TransportArgs &A, const Smem &S, int gw, int w, int type,
                                     float x, float y, float z, float ux, float uy, float uz,
                                     uint32_t E, const Lane &parent, uint32_t j) {
    uint32_t lo, hi;
    const RoundKeys<ONE> key{A, S.plans[parent.plan]};
    child_lineage(parent, j, key, lo, hi);
    const PhiloxLineage lin = philox_lineage(lo, hi, key(0), key(1));
    const unsigned slot = atomicAdd(&S.ws[w].stk[type], 1u);
    Rec *r = A.stacks + ((size_t)gw * 2 + type) * A.stack_cap + slot;
    r->a = make_float4(x, y, z, ux);
    r->b = make_float4(uy, uz, __uint_as_float(E), __uint_as_float(parent.hist));
    r->c = make_uint4(lin.a, lin.c, 0u, parent.plan);
    count(S, w, type == 0 ? CNT_PHOTONS : CNT_ELECTRONS);
}

// An electron set in motion by a photon: pushed for transport, or, in the
// photon-only mode (GPUMCD_LAUNCH_KERMA), deposited in the voxel `idx` of the
// photon's interaction.
template <bool KERMA, bool ONE>
__device__ __forceinline__ void emit_electron(const TransportArgs &A, const Smem &S, int gw, int w,
                                              const PlanDev &P, uint32_t idx, float vx, float vy, float vz,
                                              uint32_t E, const Lane &parent, uint32_t j) {
    if (KERMA)
        deposit(P, parent.hist, idx, E);
    else
        push<ONE>(A, S, gw, w, 1, parent.x, parent.y, parent.z, vx, vy, vz, E, parent, j);
}

template <bool ONE>
__device__ __forceinline__ void load_rec(const TransportArgs &A, const Smem &S, Lane &p, const Rec &r) {
    const float4 a = r.a;
    const float4 b = r.b;
    const uint4 c = r.c;
    p.x = a.x; p.y = a.y; p.z = a.z; p.ux = a.w;
    p.uy = b.x; p.uz = b.y; p.E = __float_as_uint(b.z); p.hist = __float_as_uint(b.w);
    // the plan field indexes the CTA's 64-entry plan table, all of whose
    // entries are set at launch: masked, it stays in range by construction
    p.draw = c.z; p.plan = c.w & (GPUMCD_MAX_PLANS_PER_RUN - 1);
    p.lin.a = c.x;
    p.lin.b = philox_lineage_b(c.y, RoundKeys<ONE>{A, S.plans[p.plan]}(1));
    p.lin.c = c.y;
    p.act = true;
}

__device__ __forceinline__ Rec make_rec(const Lane &p) {
    Rec r;
    r.a = make_float4(p.x, p.y, p.z, p.ux);
    r.b = make_float4(p.uy, p.uz, __uint_as_float(p.E), __uint_as_float(p.hist));
    r.c = make_uint4(p.lin.a, p.lin.c, p.draw, p.plan);
    return r;
}

// ---------------------------------------------------------------------------
// Samplers (exact, FP32)
// ---------------------------------------------------------------------------

// Klein-Nishina (GPUMCD §II.A, Compton): composition-rejection on eps = k'/k
// in [1/(1+2k), 1]: choose 1/eps or eps by their integrals, accept with
// 1 - eps sin^2 / (1 + eps^2).  Returns eps, with cos theta in *c and the
// fourth word of the last draw in *w4.
constexpr int SAMPLER_CAP = 4096;  // proposals before a sampler gives up (counted, never expected)

template <class Keys>
__device__ float sample_kn(Lane &p, const Keys &P, float k, float *c, uint32_t *w4, unsigned *capped) {
    const float e0 = __fdividef(1.0f, 1.0f + 2.0f * k);
    const float a1 = __logf(1.0f + 2.0f * k);
    const float a2 = 0.5f * (1.0f - e0 * e0);
    for (int it = 0;; ++it) {
        const uint4 r = draw4(p, P);
        float eps;
        if (u01(r.x) * (a1 + a2) < a1)
            eps = __expf(-a1 * u01(r.y));
        else
            eps = sqrtf(fmaf(1.0f - e0 * e0, u01(r.y), e0 * e0));
        const float t = __fdividef(1.0f - eps, k * eps);
        const float s2 = t * (2.0f - t);
        const bool ok = u01(r.z) <= 1.0f - __fdividef(eps * s2, 1.0f + eps * eps);
        if (ok || it >= SAMPLER_CAP) {
            if (!ok) ++*capped;
            *c = 1.0f - t;
            *w4 = r.w;
            return eps;
        }
    }
}

// Sauter photo-electron polar angle (§II.A): nu = 1 - cos drawn from
// nu/(A+nu)^3 and accepted with (2-nu)(1/(A+nu)+B) / (2(1/A+B)).
template <class Keys>
__device__ float sample_sauter(Lane &p, const Keys &P, float T, uint32_t *w3, unsigned *capped) {
    const float g = 1.0f + T / kMC2f;
    const float b2 = 1.0f - __fdividef(1.0f, g * g);
    const float beta = sqrtf(b2);
    const float A = __fdividef(__fdividef(1.0f, g * g * (1.0f + beta)), beta);
    const float B = 0.5f * beta * g * (g - 1.0f) * (g - 2.0f);
    const float gmax = 2.0f * (__fdividef(1.0f, A) + B);
    for (int it = 0;; ++it) {
        const uint4 r = draw4(p, P);
        const float sq = sqrtf(u01(r.x));
        const float nu = __fdividef(2.0f * A * sq, A + 2.0f - 2.0f * sq);
        const bool ok = u01(r.y) * gmax <= (2.0f - nu) * (__fdividef(1.0f, A + nu) + B);
        if (ok || it >= SAMPLER_CAP) {
            if (!ok) ++*capped;
            *w3 = r.z;
            return 1.0f - nu;
        }
    }
}

// Hard electron event (§II.B.1).  Moller: the knock-on fraction in [thr/T, 1/2]
// by a 1/eps^2 proposal (thr = t_c).  Bremsstrahlung: the photon energy in
// [thr, T] by a 1/k proposal (thr = k_c), accepted with the normalised shape
// (4/3 - 4y/3 + y^2) cA + (1 - y) cB.  One loop serves both, so the lanes of a
// warp share each proposal's draw (ten Philox rounds, most of a proposal)
// whichever kind they sample.
template <class Keys>
__device__ __forceinline__ float sample_hard(Lane &p, const Keys &P, bool moller, float T, float thr, float cA,
                                             float cB, uint32_t *w3, unsigned *capped) {
    float v0, v1, v2, v3;  // Moller: thr / T, c1, c2, bound; bremsstrahlung: E, ln(T / thr), cA, cB
    if (moller) {
        const float g = T / kMC2f + 1.0f;
        v0 = __fdividef(thr, T);
        v1 = __fdividef((g - 1.0f) * (g - 1.0f), g * g);
        v2 = __fdividef(2.0f * g - 1.0f, g * g);
        v3 = 2.0f + 0.25f * v1;
    } else {
        v0 = T + kMC2f;
        v1 = __logf(__fdividef(T, thr));
        v2 = cA;
        v3 = cB;
    }
    for (int it = 0;; ++it) {
        const uint4 r = draw4(p, P);
        float x;
        bool ok;
        if (moller) {
            x = __fdividef(v0, 1.0f - u01(r.x) * (1.0f - 2.0f * v0));
            const float q = __fdividef(x, 1.0f - x);
            const float f = 1.0f + q * q + v1 * x * x - v2 * q;
            ok = u01(r.y) * v3 <= f;
        } else {
            x = thr * __expf(u01(r.x) * v1);
            const float y = __fdividef(x, v0);
            const float gy = fmaf(y, y - 4.0f / 3.0f, 4.0f / 3.0f) * v2 + (1.0f - y) * v3;
            ok = u01(r.y) <= gy;
        }
        if (ok || it >= SAMPLER_CAP) {
            if (!ok) ++*capped;
            *w3 = r.z;
            return x;
        }
    }
}

// Multiple-scattering mu = (1 - cos)/2 after G1 transport mean free paths
// (§II.B.2 substitute): f(mu) ~ (mu + a)^-2 with a from the ln(a) table.
__device__ __forceinline__ float ms_mu(const float *tab, const Grid &gr, float g1, float z) {
    if (g1 < (float)MS_G_MIN) return 0.0f;
    if (g1 > (float)MS_G_MAX) return z;
    const float a = __expf(interp_ms(tab + TAB_MS, fmaf(__log2f(g1), gr.ms_a, gr.ms_b)));
    // at z = 1 the exact value is 1; in FP32, 1 + a rounds to 1 when a < 2^-24
    // and the quotient would be a / 0
    return fminf(__fdividef(a * z, 1.0f + a - z), 1.0f);
}

// The bin of quantile z in (0, 1]: the first with cdf[i+1] >= z.  The guide
// leaves a bin or two to search, where a search of all bins (256 of the 6
// MV-like spectrum) made eight dependent loads for the few lanes that take a
// primary at a time: the transport of 4e6 photons on the slabs takes 2.98 ms,
// 3.03 before.
__device__ __forceinline__ int spectrum_bin(const PlanDev &P, float z) {
    const float *cdf = P.spec;
    const int j = min(max((int)ceilf(z * (float)SPEC_GUIDE) - 1, 0), SPEC_GUIDE - 1);
    const uint32_t g = __ldg(reinterpret_cast<const uint32_t *>(P.spec) + 2 * (P.n_spec + 1) + j);
    int lo = (int)(g & 0xFFFFu), hi = (int)(g >> 16);
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (__ldg(cdf + mid + 1) >= z) hi = mid; else lo = mid + 1;
    }
    return lo;
}

__device__ __forceinline__ float sample_spectrum(const PlanDev &P, float z) {
    const float *cdf = P.spec;
    const float *edges = P.spec + P.n_spec + 1;
    const int lo = spectrum_bin(P, z);
    const float c0 = __ldg(cdf + lo), c1 = __ldg(cdf + lo + 1);
    const float f = c1 > c0 ? fminf(fmaxf((z - c0) / (c1 - c0), 0.f), 1.f) : 0.5f;
    const float e0 = __ldg(edges + lo), e1 = __ldg(edges + lo + 1);
    return fmaf(f, e1 - e0, e0);
}

// Primary of history h of plan P (§II.C.2 initParticle): pencil or square
// parallel beam entering through z = 0 along +z; with PHSP, a phase-space
// plan's primary is record h mod n as listed (the first draw is still taken,
// so the draw counter starts where the beams' does).  A source grouped by
// energy starts each history as an ungrouped one does: the grouping orders the
// claims (refill), not the sample.
template <bool PHSP, bool ONE>
__device__ __forceinline__ uint32_t make_primary(const TransportArgs &A, Lane &p, const PlanDev &P, uint32_t plan, uint64_t h) {
    const RoundKeys<ONE> key{A, P};
    p.hist = (uint32_t)h;
    p.lin = philox_lineage(1u, 0u, key(0), key(1));
    p.draw = 0u;
    p.plan = plan;
    const uint4 r = draw4(p, key);
    if (PHSP && P.beam == GPUMCD_BEAM_PHASE_SPACE) {
        const float4 *ps = reinterpret_cast<const float4 *>(P.spec);
        const uint32_t k = (uint32_t)(h % (unsigned long long)P.n_phsp);
        const float4 a = __ldg(ps + 2 * (size_t)k), b = __ldg(ps + 2 * (size_t)k + 1);
        p.x = a.x;
        p.y = a.y;
        p.z = a.z;
        p.ux = b.x;
        p.uy = b.y;
        p.uz = b.z;
        p.E = __float2uint_rn(a.w * kInvQf);
        p.act = true;
        return p.E;
    }
    p.x = P.cx;
    p.y = P.cy;
    if (P.beam == GPUMCD_BEAM_SQUARE) {
        p.x = fmaf(u01(r.x) - 0.5f, P.field, P.cx);
        p.y = fmaf(u01(r.y) - 0.5f, P.field, P.cy);
    }
    p.z = 0.0f;
    p.ux = 0.0f;
    p.uy = 0.0f;
    p.uz = 1.0f;
    const float zq = u01(r.z);
    p.E = P.n_spec > 0 ? __float2uint_rn(sample_spectrum(P, zq) * kInvQf) : P.e_src_q;
    p.act = true;
    return p.E;
}

// ---------------------------------------------------------------------------
// Photon transport
// ---------------------------------------------------------------------------
// Photon (GPUMCD §II.A).  photon_flight: one Woodcock flight; true when it
// ends on a real event, with its voxel, the word that picks the interaction,
// and the voxel's material, density and attenuation coefficient.  xp (the
// energy's grid coordinate) and mu_hat (the majorant) are the caller's, taken
// once for all flights of a pass: the energy does not change on a fictitious
// event.  photon_interact: that interaction (Compton, photoelectric or pair,
// by the partial attenuation coefficients of the voxel's material).
template <bool ONE>
__device__ __forceinline__ bool photon_flight(const TransportArgs &A, const Smem &S, Lane &p, float xp,
                                              float mu_hat, uint32_t &idx_out, uint32_t &rz, int &m_out,
                                              float &rho_out, float &mu_out, int w) {
    const PlanDev &P = S.plans[p.plan];
    const Phys &ph = A.phys;
    const uint4 r = draw4(p, RoundKeys<ONE>{A, P});
    const float s = __fdividef(-__logf(u01(r.x)), mu_hat);
    p.x = fmaf(s, p.ux, p.x);
    p.y = fmaf(s, p.uy, p.y);
    p.z = fmaf(s, p.uz, p.z);
    if (!inside(P, p.x, p.y, p.z)) {
        ledger_add(S, p.plan, 1, p.E);
        p.act = false;
        return false;
    }
    int ix, iy, iz;
    const uint32_t idx = voxel_index(P, p.x, p.y, p.z, ix, iy, iz);
    const uint32_t vw = __ldg(P.vox + idx);
    const int m = vw & (NMAT - 1);  // ids < NMAT (checked when packed): in range by construction
    const float rho = (float)(vw >> 4) * kRhoQ;
    const float *tp = S.tab + tab_ph(m);
    const bool pair_open = p.E > ph.two_mc2_q;
    float mu = rho * interp(tp, xp);
    if (!pair_open) mu = rho * (interp(tp + G, xp) + interp(tp + 2 * G, xp));
    if (u01(r.y) * mu_hat > mu) return false;  // fictitious: direction and energy unchanged
    count(S, w, CNT_PH_REAL);
    idx_out = idx;
    rz = r.z;
    m_out = m;
    rho_out = rho;
    mu_out = mu;
    return true;
}

template <bool KERMA, bool ONE>
__device__ __forceinline__ void photon_interact(const TransportArgs &A, const Smem &S, Lane &p, uint32_t idx,
                                                uint32_t rz, float xp, int m, float rho, float mu, int gw,
                                                int w) {
    const PlanDev &P = S.plans[p.plan];
    const Phys &ph = A.phys;
    const float *tp = S.tab + tab_ph(m);
    const bool pair_open = p.E > ph.two_mc2_q;
    const float muC = rho * interp(tp + G, xp);
    const float mupe = rho * interp(tp + 2 * G, xp);
    const float q = u01(rz) * mu;
    const float E = (float)p.E * kQf;
    if (q < muC) {
        // Compton scattering on a free electron (Klein-Nishina).
        count(S, w, CNT_COMPTON);
        float c;
        uint32_t w4;
        unsigned capped = 0;
        const float eps = sample_kn(p, RoundKeys<ONE>{A, P}, E / kMC2f, &c, &w4, &capped);
        if (capped) count(S, w, CNT_SAMPLER_CAP);
        float sp, cp;
        __sincosf(kTWO_PIf * u01(w4), &sp, &cp);
        const float sn = sqrtf(fmaxf(0.0f, (1.0f - c) * (1.0f + c)));
        const uint32_t e1 = min(p.E, __float2uint_rn(eps * (float)p.E));
        const uint32_t te = p.E - e1;
        float vx = p.ux, vy = p.uy, vz = p.uz;
        rotate(vx, vy, vz, c, sn, cp, sp);
        if (te >= ph.e_abs_q) {
            // recoil direction from momentum balance: E u - E' u'
            const float e1f = (float)e1 * kQf;
            float ex = E * p.ux - e1f * vx, ey = E * p.uy - e1f * vy, ez = E * p.uz - e1f * vz;
            const float n = rsqrtf(fmaxf(ex * ex + ey * ey + ez * ez, 1e-30f));
            emit_electron<KERMA, ONE>(A, S, gw, w, P, idx, ex * n, ey * n, ez * n, te, p, 0);
        } else {
            deposit(P, p.hist, idx, te);
        }
        p.ux = vx;
        p.uy = vy;
        p.uz = vz;
        p.E = e1;
        if (e1 < ph.p_cut_q) {
            deposit(P, p.hist, idx, e1);
            p.act = false;
        }
    } else if (q < muC + mupe || !pair_open) {
        // Photoelectric: one K-shell electron carrying all of E (no binding).
        count(S, w, CNT_PHOTO);
        if (p.E >= ph.e_abs_q) {
            uint32_t w3;
            unsigned capped = 0;
            const float c = sample_sauter(p, RoundKeys<ONE>{A, P}, E, &w3, &capped);
            if (capped) count(S, w, CNT_SAMPLER_CAP);
            float sp, cp;
            __sincosf(kTWO_PIf * u01(w3), &sp, &cp);
            const float sn = sqrtf(fmaxf(0.0f, (1.0f - c) * (1.0f + c)));
            float vx = p.ux, vy = p.uy, vz = p.uz;
            rotate(vx, vy, vz, c, sn, cp, sp);
            emit_electron<KERMA, ONE>(A, S, gw, w, P, idx, vx, vy, vz, p.E, p, 0);
        } else {
            deposit(P, p.hist, idx, p.E);
        }
        p.act = false;
    } else {
        // Pair production without positrons: two electrons share E - 2mc^2
        // uniformly, the rest energy goes to its own ledger.
        count(S, w, CNT_PAIR);
        const uint32_t tt = p.E - ph.two_mc2_q;
        ledger_add(S, p.plan, 2, ph.two_mc2_q);
        const uint4 r2 = draw4(p, RoundKeys<ONE>{A, P});
        const uint32_t t1 = min(tt, __float2uint_rn(u01(r2.x) * (float)tt));
        const uint32_t t2 = tt - t1;
        float sp, cp;
        __sincosf(kTWO_PIf * u01(r2.y), &sp, &cp);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const uint32_t te = j == 0 ? t1 : t2;
            if (te >= ph.e_abs_q) {
                const float th = __fdividef(kMC2f, (float)te * kQf + kMC2f);
                float st, ct;
                __sincosf(th, &st, &ct);
                float vx = p.ux, vy = p.uy, vz = p.uz;
                rotate(vx, vy, vz, ct, st, j == 0 ? cp : -cp, j == 0 ? sp : -sp);
                emit_electron<KERMA, ONE>(A, S, gw, w, P, idx, vx, vy, vz, te, p, (uint32_t)j);
            } else {
                deposit(P, p.hist, idx, te);
            }
        }
        p.act = false;
    }
}

// ---------------------------------------------------------------------------
// Electron: one condensed-history step (GPUMCD §II.B.3)
// ---------------------------------------------------------------------------
// The energy lost along the step is not deposited here: its voxel and amount
// come back in dep_idx / dep_e so the caller can deposit it at a convergent
// point.  The particle starts inside the phantom, so its voxel index is in
// range: electron primaries are tested when they are claimed, secondaries
// start at interaction points inside, and a step that ends outside ends the
// particle.  It starts above the absorption energy (the caller tests it).  A
// step that ends outside or below that energy sets fin and leaves the end
// point and the energy in p, for electron_end.
template <bool ONE>
__device__ __forceinline__ void electron_step(const TransportArgs &A, const Smem &S, Lane &p, int gw, int w,
                                              uint32_t &dep_idx, uint32_t &dep_e, bool &fin) {
    const PlanDev &P = S.plans[p.plan];
    const Phys &ph = A.phys;
    int ix, iy, iz;
    const uint32_t idx0 = voxel_index(P, p.x, p.y, p.z, ix, iy, iz);
    const uint32_t vw = __ldg(P.vox + idx0);
    // the step's draw, taken while the voxel word is on its way
    const uint4 r = draw4(p, RoundKeys<ONE>{A, P});
    const int m0 = vw & (NMAT - 1);
    const float rho0 = (float)(vw >> 4) * kRhoQ;
    const float *te = S.tab + tab_el(m0);
    const float T = (float)p.E * kQf;
    const float xe = fmaf(__log2f((float)p.E), ph.grid.el_a, ph.grid.el_bq);
    const float L0 = rho0 * interp(te, xe);
    const float smax = __fdividef(ph.estepe * T, L0);
    // distance to the voxel faces along u, plus the nudge
    float dv = exit_distance(P, p, ix, iy, iz);
    dv = fmaxf(dv, 0.0f) + ph.nudge;
    // The step stays in its voxel (it ends at the exit face, plus the nudge),
    // so the voxel's own hard cross-section at the start energy bounds it over
    // the step: Sigma_hard,m rises with T, and T only falls along the step.
    // The margin covers the rounding of the two interpolations.
    const float sig_hat = rho0 * interp(te + G, xe) * kHardMajorantMargin;
    const float ehard = __fdividef(-__logf(u01(r.x)), sig_hat);
    float es = fminf(dv, smax);
    const bool hard = ehard < es;
    es = fminf(es, ehard);
    // Delta E = e_s L(E0 - L(E0) e_s / 2)
    const float tm = fmaxf(T - 0.5f * L0 * es, 1e-6f);
    const float dE = es * rho0 * interp(te, fmaf(__log2f(tm), ph.grid.el_a, ph.grid.el_bm));
    const uint32_t dq = min(p.E, __float2uint_rn(dE * kInvQf));
    const uint32_t e1 = p.E - dq;
    // random hinge: move z e_s, deflect with the energy before or after the
    // loss (coin from the low bit of the first word), deposit, move (1 - z) e_s
    const float zh = u01(r.y);
    const float l1 = zh * es;
    float x = fmaf(l1, p.ux, p.x), y = fmaf(l1, p.uy, p.y), z = fmaf(l1, p.uz, p.z);
    const float tms = fmaxf((r.x & 1u) ? T : (float)e1 * kQf, 1e-6f);
    const float g1 = es * rho0 * interp(te + 3 * G, fmaf(__log2f(tms), ph.grid.el_a, ph.grid.el_bm));
    const float mu = ms_mu(S.tab, ph.grid, g1, u01(r.z));
    if (mu > 0.0f) {
        float sp, cp;
        __sincosf(kTWO_PIf * u01(r.w), &sp, &cp);
        rotate(p.ux, p.uy, p.uz, 1.0f - 2.0f * mu, 2.0f * sqrtf(mu * (1.0f - mu)), cp, sp);
    }
    dep_idx = idx0;  // the hinge lies in the step-start voxel
    dep_e = dq;
    const float l2 = es - l1;
    // each coordinate one float further along the direction (float_along)
    p.x = float_along(fmaf(l2, p.ux, x), p.ux);
    p.y = float_along(fmaf(l2, p.uy, y), p.uy);
    p.z = float_along(fmaf(l2, p.uz, z), p.uz);
    p.E = e1;
    if (e1 < ph.e_abs_q || !inside(P, p.x, p.y, p.z)) {
        p.act = false;
        fin = true;
        return;
    }
    if (!hard) return;
    // A hard-event candidate: park the particle for a converged hard pass of
    // its warp (the candidate test and the event follow there, with the same
    // random draws in the same order, so the result does not change).
    {
        const unsigned slot = atomicAdd(&S.ws[w].hc, 1u);
        HardRec &h = A.hard[(size_t)gw * HARD_CAP + slot];
        h.r = make_rec(p);
        h.sig_hat = sig_hat;
        h.idx = idx0;
        p.act = false;
    }
}

// An electron at the end of its path: absorbed where it is, or escaped.
__device__ __forceinline__ void electron_end(const Smem &S, const Lane &p) {
    const PlanDev &P = S.plans[p.plan];
    if (inside(P, p.x, p.y, p.z)) {
        int ix, iy, iz;
        deposit(P, p.hist, voxel_index(P, p.x, p.y, p.z, ix, iy, iz), p.E);
    } else {
        ledger_add(S, p.plan, 1, p.E);
    }
}

// ---------------------------------------------------------------------------
// Electron hard event (GPUMCD §II.B.3): the electron Woodcock test at the end
// of a step whose sampled hard distance was the shortest, then Moller or
// bremsstrahlung.  Runs in the warp's hard pass with the parked candidate in
// the lane: p after its step, sig_hat = the step's majorant, idx1 = the step's
// voxel, which holds the candidate point (the step ends inside it, or at most
// the nudge past its face) and so the event and its sub-cut-off deposits.
// ---------------------------------------------------------------------------
template <bool ONE>
__device__ __forceinline__ void hard_event(const TransportArgs &A, const Smem &S, Lane &p, float sig_hat,
                                        uint32_t idx1, int gw, int w) {
    const PlanDev &P = S.plans[p.plan];
    const Phys &ph = A.phys;
    const uint32_t e1 = p.E;
    // electron Woodcock: accept a real hard event with Sigma(T_end)/Sigma_hat
    const uint32_t vw1 = __ldg(P.vox + idx1);
    const uint4 r2 = draw4(p, RoundKeys<ONE>{A, P});  // the event's draw, taken while the voxel word loads
    const int m1 = vw1 & (NMAT - 1);
    const float rho1 = (float)(vw1 >> 4) * kRhoQ;
    const float *t1 = S.tab + tab_el(m1);
    const float xe1 = fmaf(__log2f((float)e1), ph.grid.el_a, ph.grid.el_bq);
    const float T1 = (float)e1 * kQf;
    // Moller needs T > 2 t_c and bremsstrahlung T > k_c (zero below, as in the
    // closed forms; the interpolated tables are not exactly zero there)
    const float sb = T1 > ph.k_c ? rho1 * interp(t1 + 2 * G, xe1) : 0.0f;
    const float sm = T1 > 2.0f * ph.t_c ? fmaxf(rho1 * interp(t1 + G, xe1) - sb, 0.0f) : 0.0f;
    const float sig = sm + sb;
    if (u01(r2.x) * sig_hat >= sig) {
        count(S, w, CNT_HARD_FICT);
        return;
    }
    count(S, w, CNT_HARD_REAL);
    const bool moller = u01(r2.y) * sig < sm;
    count(S, w, moller ? CNT_MOLLER : CNT_BREM);
    // The two kinds share the proposals' draws, the azimuth, the rotation and
    // the push of the new particle.  As two branches, each ran its own copy
    // with its part of the lanes (about two thirds Moller): 15 MeV electrons
    // on 128^3 water took 1.85 ms of transport, 1.77 this way, photons 4.19
    // and 4.09.
    uint32_t w3;
    unsigned capped = 0;
    const float x = sample_hard(p, RoundKeys<ONE>{A, P}, moller, T1, moller ? ph.t_c : ph.k_c, S.tab[TAB_BREM + 2 * m1],
                                S.tab[TAB_BREM + 2 * m1 + 1], &w3, &capped);
    if (capped) count(S, w, CNT_SAMPLER_CAP);
    uint32_t e2;
    float c, sn, c2 = 1.0f;
    if (moller) {
        // knock-on and scattered electron, azimuths phi and phi + pi
        e2 = min(e1, __float2uint_rn(x * (float)e1));
        const uint32_t tp = e1 - e2;
        const float tkf = (float)e2 * kQf, tpf = (float)tp * kQf;
        c = sqrtf(fminf(1.0f, __fdividef(tkf * (T1 + 2.0f * kMC2f), T1 * (tkf + 2.0f * kMC2f))));
        c2 = sqrtf(fminf(1.0f, __fdividef(tpf * (T1 + 2.0f * kMC2f), T1 * (tpf + 2.0f * kMC2f))));
        sn = sqrtf(fmaxf(0.f, 1.f - c * c));
    } else {
        // electron direction kept, photon at theta = mc^2/E
        e2 = min(e1, __float2uint_rn(x * kInvQf));
        __sincosf(__fdividef(kMC2f, T1 + kMC2f), &sn, &c);
    }
    float sp, cp;
    __sincosf(kTWO_PIf * u01(w3), &sp, &cp);
    float vx = p.ux, vy = p.uy, vz = p.uz;
    rotate(vx, vy, vz, c, sn, cp, sp);
    if (e2 >= (moller ? ph.e_abs_q : ph.p_cut_q))
        push<ONE>(A, S, gw, w, moller ? 1 : 0, p.x, p.y, p.z, vx, vy, vz, e2, p, 0);
    else
        deposit(P, p.hist, idx1, e2);
    if (moller) rotate(p.ux, p.uy, p.uz, c2, sqrtf(fmaxf(0.f, 1.f - c2 * c2)), -cp, -sp);
    p.E = e1 - e2;
}

// ---------------------------------------------------------------------------
// Warp scheduling helpers (all called by the whole warp, convergent)
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned lanemask_lt() {
    unsigned m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Claim records of a global source of type t with a cursor and a fixed count:
// `chunk` of them while there is plenty, fewer so that every warp gets a share.
// A photon source shorter than a chunk per warp is split evenly.  Of an
// electron source a warp takes an even share of what is left, so the claims
// shrink towards the end: an electron's path is a chain of tens of steps that
// nothing shortens, so late claims of 32 left some warps a full load to run
// while the others had ended.  Transport against claims of 32 throughout: 3001
// electrons of 9 MeV 0.31 -> 0.18 ms, 1e4 photons of 2 MeV 0.125 -> 0.084 ms,
// 1e6 electrons of 15 MeV 1.94 -> 1.83 ms; no case is slower.  Shrinking
// claims of photons cost 4e6 of 15 MeV 3.5% (4.22 -> 4.37 ms) and the slab
// plan 1.6%: photon warps then run half empty and switch type more often.
__device__ __forceinline__ void claim(unsigned long long *cursor, unsigned long long total, uint32_t chunk, int t,
                                      unsigned long long &lo, unsigned long long &hi) {
    const uint32_t warps = gridDim.x * (blockDim.x >> 5);
    unsigned long long left = total;
    if (t == 1) {
        const unsigned long long now = *(volatile unsigned long long *)cursor;
        left = now < total ? total - now : 0ull;
    }
    const uint32_t want = left >= (unsigned long long)chunk * warps ? chunk : max((uint32_t)left / warps, 1u);
    const unsigned long long base = atomicAdd(cursor, (unsigned long long)want);
    lo = base < total ? base : total;
    hi = base + want < total ? base + want : total;
}

// Per-CTA flags that remember exhausted global sources, so a warp does not
// re-read global counters once a source is known to be empty.
struct CtaFlags {
    int in_done[2];
    int prim_done[2];
};

// Shared memory of a CTA: the plan table, warp states, counters, ledgers, the
// mbarrier and the source flags (fixed size, rounded up to 128 bytes), then the
// tables staged by the bulk copy.
constexpr size_t SMEM_FIXED = (sizeof(PlanDev) * GPUMCD_MAX_PLANS_PER_RUN + sizeof(WarpState) * MAX_WARPS +
                               sizeof(unsigned int) * MAX_WARPS * CNT_ROW +
                               sizeof(unsigned long long) * (CNT_N + 3 * GPUMCD_MAX_PLANS_PER_RUN + 1) +
                               sizeof(CtaFlags) + 127) / 128 * 128;
// Three CTAs stay resident (block_threads <= 256 with blocks_per_sm = 3) with
// every material loaded: an SM has 228 KB, of which each CTA takes 1 KB besides.
// With counter rows of all CNT_N words only two did: 256 x 3 took 2.37 ms for 1e6
// electrons of 15 MeV and 2.92 for 2e6 photons on 128^3 water, 2.10 and 2.54 so.
static_assert(3 * (SMEM_FIXED + TAB_BYTES + 1024) <= 228 * 1024, "three CTAs of all materials");

// Move the top n records of stack `t` to the global overflow queue.  A full
// queue sets GPUMCD_ERR_QUEUE_OVERFLOW: the run is then invalid and reported,
// never silently truncated.
__device__ void spill_to_queue(const TransportArgs &A, const Smem &S, int gw, int w, int t, unsigned n) {
    const int lane = threadIdx.x & 31;
    const unsigned top = S.ws[w].stk[t];
    n = min(n, top);
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(A.out[t].cursor, (unsigned long long)n);
    base = __shfl_sync(FULL, base, 0);
    const Rec *src = A.stacks + ((size_t)gw * 2 + t) * A.stack_cap + (top - n);
    for (unsigned i = lane; i < n; i += 32)
        if (base + i < A.out[t].capacity) A.out[t].rec[base + i] = src[i];
    if (lane == 0) {
        if (base + n > A.out[t].capacity) {
            atomicExch(A.error, GPUMCD_ERR_QUEUE_OVERFLOW);
            count(S, w, CNT_OVERFLOW);
        }
        S.ws[w].stk[t] = top - n;
        atomicAdd(counter(S, w, CNT_SPILLS), n);
    }
    __syncwarp();
}

// Fill empty lanes with particles of type t.  Returns the number of lanes
// that hold a particle afterwards.
template <bool KERMA, bool PHSP, bool ONE>
__device__ int refill(const TransportArgs &A, const Smem &S, CtaFlags &F, Lane &p, int gw, int w, int t) {
    const int lane = threadIdx.x & 31;
    WarpState &ws = S.ws[w];
    unsigned empty = __ballot_sync(FULL, !p.act);
    if (empty == 0u) return 32;
    const unsigned lt = lanemask_lt();
    // 1) the warp's private stack (newest first)
    {
        const unsigned sc = ws.stk[t];
        const unsigned take = min((unsigned)__popc(empty), sc);
        if (take) {
            const unsigned rank = __popc(empty & lt);
            if (!p.act && rank < take)
                load_rec<ONE>(A, S, p, A.stacks[((size_t)gw * 2 + t) * A.stack_cap + (sc - 1u - rank)]);
            __syncwarp();
            if (lane == 0) ws.stk[t] = sc - take;
            __syncwarp();
            empty = __ballot_sync(FULL, !p.act);
            if (empty == 0u) return 32;
        }
    }
    // 2) the overflow queue of the previous launch, in chunks
    for (int pass = 0; pass < 2; ++pass) {
        unsigned long long lo = ws.q_lo[t], hi = ws.q_hi[t];
        if (lo == hi) {
            if (__shfl_sync(FULL, lane == 0 ? *(volatile int *)&F.in_done[t] : 0, 0)) break;
            if (lane == 0) claim(A.in[t].cursor, A.in_count[t], A.chunk, t, lo, hi);
            lo = __shfl_sync(FULL, lo, 0);
            hi = __shfl_sync(FULL, hi, 0);
            if (lo == hi) {
                if (lane == 0) F.in_done[t] = 1;
                break;
            }
        }
        const unsigned take = (unsigned)min((unsigned long long)__popc(empty), hi - lo);
        const unsigned rank = __popc(empty & lt);
        if (!p.act && rank < take) load_rec<ONE>(A, S, p, A.in[t].rec[lo + rank]);
        __syncwarp();
        if (lane == 0) {
            ws.q_lo[t] = lo + take;
            ws.q_hi[t] = hi;
        }
        __syncwarp();
        empty = __ballot_sync(FULL, !p.act);
        if (empty == 0u) return 32;
    }
    // 3) primaries of this type, in chunks
    for (int pass = 0; pass < 2; ++pass) {
        unsigned long long lo = ws.p_lo[t], hi = ws.p_hi[t];
        if (lo == hi) {
            if (__shfl_sync(FULL, lane == 0 ? *(volatile int *)&F.prim_done[t] : 0, 0)) break;
            if (lane == 0) claim(&A.prim_cursor[t], A.prim_off[t][A.n_prim_plans[t]], A.chunk, t, lo, hi);
            lo = __shfl_sync(FULL, lo, 0);
            hi = __shfl_sync(FULL, hi, 0);
            if (lo == hi) {
                if (lane == 0) F.prim_done[t] = 1;
                break;
            }
        }
        const unsigned take = (unsigned)min((unsigned long long)__popc(empty), hi - lo);
        const unsigned rank = __popc(empty & lt);
        if (!p.act && rank < take) {
            const unsigned long long g = lo + rank;
            int a = 0, b = (int)A.n_prim_plans[t] - 1;  // last plan with prim_off <= g
            while (a < b) {
                const int mid = (a + b + 1) >> 1;
                if (A.prim_off[t][mid] <= g) a = mid; else b = mid - 1;
            }
            const uint32_t plan = A.prim_plan[t][a];
            const PlanDev &P = S.plans[plan];
            unsigned long long j = g - A.prim_off[t][a];
            // a source grouped by energy: its histories are claimed in
            // decreasing order of their energy (the order its launch sorted)
            if (PHSP && P.e_group && j < P.n_sorted) j = __ldg(P.order + j);
            ledger_add(S, plan, 0, make_primary<PHSP, ONE>(A, p, P, plan, P.hist_base + j));
            if (t == 0 && p.E < A.phys.p_cut_q) {
                // a photon primary below the photon cut-off deposits where it
                // starts, or escapes from outside (every other photon flies
                // above the cut-off)
                if (inside(P, p.x, p.y, p.z)) {
                    int ix, iy, iz;
                    deposit(P, p.hist, voxel_index(P, p.x, p.y, p.z, ix, iy, iz), p.E);
                } else {
                    ledger_add(S, plan, 1, p.E);
                }
                p.act = false;
            }
            if (!KERMA && t == 1 && !inside(P, p.x, p.y, p.z)) {
                // an electron primary aimed outside the phantom escapes at once
                // (every other electron starts its steps inside)
                ledger_add(S, plan, 1, p.E);
                p.act = false;
            }
            if (KERMA && t == 1) {
                // photon-only mode: a primary electron deposits where it enters
                if (inside(P, p.x, p.y, p.z)) {
                    int ix, iy, iz;
                    deposit(P, p.hist, voxel_index(P, p.x, p.y, p.z, ix, iy, iz), p.E);
                } else {
                    ledger_add(S, plan, 1, p.E);
                }
                p.act = false;
            }
        }
        __syncwarp();
        if (lane == 0) {
            ws.p_lo[t] = lo + take;
            ws.p_hi[t] = hi;
            atomicAdd(counter(S, w, t == 0 ? CNT_PHOTONS : CNT_ELECTRONS), take);
        }
        __syncwarp();
        empty = __ballot_sync(FULL, !p.act);
        if (empty == 0u) return 32;
    }
    return 32 - __popc(empty);
}

// Particles of type t the warp could still take (a global source counts 32).
// Evaluated by lane 0 and broadcast, so the whole warp takes the same branch.
__device__ __forceinline__ unsigned available(const TransportArgs &A, const Smem &S, CtaFlags &F, int w,
                                              int t) {
    unsigned n = 0;
    if ((threadIdx.x & 31) == 0) {
        const WarpState &ws = S.ws[w];
        n = ws.stk[t] + (t == 1 ? ws.hc : 0u);  // parked hard candidates are electrons
        if (ws.q_lo[t] < ws.q_hi[t]) n += 32;
        else if (!*(volatile int *)&F.in_done[t]) {
            if (*(volatile unsigned long long *)A.in[t].cursor < A.in_count[t]) n += 32;
            else F.in_done[t] = 1;
        }
        if (ws.p_lo[t] < ws.p_hi[t]) n += 32;
        else if (!*(volatile int *)&F.prim_done[t]) {
            if (*(volatile unsigned long long *)&A.prim_cursor[t] < A.prim_off[t][A.n_prim_plans[t]]) n += 32;
            else F.prim_done[t] = 1;
        }
    }
    return __shfl_sync(FULL, n, 0);
}

// The warp's hard pass: park its stepping electrons on their stack, take up
// to 32 parked hard-event candidates into the lanes and run their events
// together.  The lanes then hold electrons again (after their events), so
// the warp goes on stepping electrons.
template <bool ONE>
__device__ __forceinline__ void hard_pass(const TransportArgs &A, const Smem &S, Lane &p, int gw, int w) {
    const int lane = threadIdx.x & 31;
    if (S.ws[w].stk[1] + 32u > A.stack_cap) spill_to_queue(A, S, gw, w, 1, 64u);
    const unsigned actm = __ballot_sync(FULL, p.act);
    const unsigned base = S.ws[w].stk[1];
    if (p.act) {
        const unsigned rank = __popc(actm & lanemask_lt());
        A.stacks[((size_t)gw * 2 + 1) * A.stack_cap + base + rank] = make_rec(p);
        p.act = false;
    }
    __syncwarp();
    const unsigned hc = S.ws[w].hc;
    const unsigned take = min(32u, hc);
    float sig_hat = 0.f;
    uint32_t idx1 = 0u;
    if ((unsigned)lane < take) {
        const HardRec &h = A.hard[(size_t)gw * HARD_CAP + (hc - 1u - lane)];
        load_rec<ONE>(A, S, p, h.r);
        sig_hat = h.sig_hat;
        idx1 = h.idx;
    }
    __syncwarp();
    if (lane == 0) {
        S.ws[w].stk[1] = base + __popc(actm);
        S.ws[w].hc = hc - take;
        count(S, w, CNT_HARD_PASSES);
    }
    __syncwarp();
    // headroom for the events' secondaries (at most one per lane per type)
    if (S.ws[w].stk[0] + 64u > A.stack_cap) spill_to_queue(A, S, gw, w, 0, 64u);
    if (S.ws[w].stk[1] + 64u > A.stack_cap) spill_to_queue(A, S, gw, w, 1, 64u);
    if (p.act) hard_event<ONE>(A, S, p, sig_hat, idx1, gw, w);
    __syncwarp();
}

// Woodcock flights a photon takes in one pass while its events are fictitious.
// Four against three: 0.3-0.9% less transport time on the density fields, the
// slabs and the 15 MeV photon beam, 4.5% less on 3001 electrons, none slower;
// five cost the slabs 1.2%.
constexpr int PH_FLIGHTS = 4;

// Condensed-history steps an electron warp takes before it refills its lanes.
// A step is about 400 warp-instructions, and going back for the refill, the
// parked-candidate, switch and headroom tests some 250 more; about a sixth of
// the lanes park a hard candidate or end in a step.  So a warp goes back only
// once a quarter of its lanes is empty, and settles the electrons that ended
// (electron_end) then, together.  Measured, transport of 1e6 15 MeV electrons
// on 128^3 water: 2.14 ms with a refill after every step, 2.00 at two or three
// steps whatever the lanes, 1.98 at four steps and a quarter empty (2.00 at a
// sixth or a third), 1.94 with the ends settled after the steps.  A lane parks
// once at most between refills, so HARD_CAP holds as with one step.
constexpr int EL_STEPS = 4;

// ---------------------------------------------------------------------------
// The kernel
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

// PROF compiles in the per-type cycle profile (GPUMCD_LAUNCH_PROFILE), AGG
// the warp-aggregated deposit (GPUMCD_LAUNCH_WARP_AGGREGATE), SCHED the
// refill policies of the divergence-reduction ablation (refill_period != 1),
// KERMA the photon-only mode (GPUMCD_LAUNCH_KERMA), PHSP phase-space sources
// and ONE launches of one plan; the production instantiations carry none of
// the first five.
template <int MAXT, int MINB, bool PROF, bool AGG, bool SCHED, bool KERMA, bool PHSP, bool ONE>
__global__ void __launch_bounds__(MAXT, MINB) k_transport(const __grid_constant__ TransportArgs A) {
    // the fixed-size parts first, at offsets known at compile time; the tables
    // of the loaded materials after them
    extern __shared__ __align__(128) unsigned char smem_raw[];
    PlanDev *plans = (PlanDev *)smem_raw;
    WarpState *ws = (WarpState *)(plans + GPUMCD_MAX_PLANS_PER_RUN);
    unsigned int *wcnt = (unsigned int *)(ws + MAX_WARPS);
    unsigned long long *cnt = (unsigned long long *)(wcnt + MAX_WARPS * CNT_ROW);
    unsigned long long *ledger = cnt + CNT_N;
    unsigned long long *mbar = ledger + 3 * GPUMCD_MAX_PLANS_PER_RUN;
    CtaFlags *flags = (CtaFlags *)(mbar + 1);
    float *tab = (float *)(smem_raw + SMEM_FIXED);

    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int gw = blockIdx.x * (blockDim.x >> 5) + w;

    // Stage the material tables into shared memory with one bulk (TMA) copy
    // completed on an mbarrier; the other threads set up the rest meanwhile.
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(mbar)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(mbar)),
                     "r"(A.tab_bytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                smem_addr(tab)),
            "l"(A.tables), "r"(A.tab_bytes), "r"(smem_addr(mbar))
            : "memory");
    }
    // every entry is set (unused ones copy plan 0), so any masked plan index
    // a record carries reaches valid pointers
    for (int i = tid; i < GPUMCD_MAX_PLANS_PER_RUN; i += blockDim.x) plans[i] = A.plans[i < A.n_plans ? i : 0];
    for (int i = tid; i < MAX_WARPS; i += blockDim.x) {
        ws[i].stk[0] = ws[i].stk[1] = 0;
        ws[i].hc = 0;
        ws[i].p_lo[0] = ws[i].p_hi[0] = ws[i].p_lo[1] = ws[i].p_hi[1] = 0;
        ws[i].q_lo[0] = ws[i].q_hi[0] = ws[i].q_lo[1] = ws[i].q_hi[1] = 0;
    }
    for (int i = tid; i < MAX_WARPS * CNT_ROW; i += blockDim.x) wcnt[i] = 0u;
    for (int i = tid; i < CNT_N + 3 * GPUMCD_MAX_PLANS_PER_RUN; i += blockDim.x) cnt[i] = 0;
    if (tid < 2) {
        flags->in_done[tid] = A.in_count[tid] == 0;
        flags->prim_done[tid] = A.prim_off[tid][A.n_prim_plans[tid]] == 0;
    }
    __syncthreads();  // also orders the mbarrier init before the waits below
    uint32_t done = 0;
    for (uint32_t it = 0; it < (1u << 26) && !done; ++it) {
        asm volatile(
            "{ .reg .pred p; mbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0; selp.u32 %0, 1, 0, p; }"
            : "=r"(done)
            : "r"(smem_addr(mbar))
            : "memory");
    }
    if (__syncthreads_or(!done)) {
        // The table copy did not complete within the bound: report it and
        // leave without touching the tables.
        if (tid == 0) atomicExch(A.error, GPUMCD_ERR_TIMEOUT);
        return;
    }
    const Smem S{tab, plans, ws, wcnt, cnt, (unsigned int *)ledger};
    CtaFlags &F = *flags;

    Lane p;
    p.act = false;
    p.x = p.y = p.z = p.ux = p.uy = p.uz = 0.f;
    p.E = p.hist = p.draw = p.plan = 0;
    p.lin = PhiloxLineage{0u, 0u, 0u};
    constexpr bool agg = AGG;
    constexpr bool prof = PROF;
    // start on the type that has work (electron-beam launches start on electrons)
    int t = available(A, S, F, w, 1) > available(A, S, F, w, 0) ? 1 : 0;
    unsigned iter = 0;
    for (;;) {
        __syncwarp();
        if ((++iter & 255u) == 0u) {
            int err = 0;
            if (lane == 0) err = *(volatile int *)A.error;
            if (__shfl_sync(FULL, err, 0) != 0) break;
            if (iter >= (1u << 24)) {
                if (lane == 0) atomicExch(A.error, GPUMCD_ERR_TIMEOUT);
                break;
            }
        }
        long long c0 = prof ? clock64() : 0;
        int n_act;
        bool fresh = true;  // this pass refilled the lanes
        if (SCHED && A.refill_period != 1u) {
            // the ablation's refill policies (GPUMCD §II.C.3): empty lanes wait
            // for every N-th pass, for the whole warp to empty, or not at all
            const unsigned actm = __ballot_sync(FULL, p.act);
            const bool wait = A.refill_period == GPUMCD_REFILL_WHEN_EMPTY ||
                              (A.refill_period != GPUMCD_REFILL_EVERY_PASS && iter % A.refill_period != 0u);
            if (actm != 0u && wait) {
                n_act = __popc(actm);
                fresh = false;
            } else {
                n_act = refill<KERMA, PHSP, ONE>(A, S, F, p, gw, w, t);
            }
        } else {
            n_act = refill<KERMA, PHSP, ONE>(A, S, F, p, gw, w, t);
        }
        if (prof && lane == 0) atomicAdd(&S.cnt[CNT_PROF_REFILL_CYC], (unsigned long long)(clock64() - c0));
        const int o = 1 - t;
        // electrons: a converged hard pass once 32 candidates are parked (each
        // lane parks at most one more before the next refill, within HARD_CAP), or sooner when the
        // warp has few electrons left to step
        if (t == 1) {
            const unsigned hc = S.ws[w].hc;
            // With few electrons left (the drain), a pass runs once the parked
            // candidates outnumber the stepping electrons, not at every
            // iteration; n_act == 0 keeps parked candidates from being left
            // behind (also when refill_low is 0).
            if (hc >= 32u || (hc > 0u && (n_act == 0 || (n_act < (int)A.refill_low && hc >= (unsigned)n_act)))) {
                hard_pass<ONE>(A, S, p, gw, w);
                continue;
            }
        }
        if (n_act == 0) {
            if (available(A, S, F, w, o) > 0u) {
                t = o;
                continue;
            }
            break;  // nothing left of either type for this warp
        }
        const unsigned so = S.ws[w].stk[o], st = S.ws[w].stk[t];
        if ((so >= A.switch_high && so > st + 32u) ||
            (n_act < (int)A.refill_low && fresh && available(A, S, F, w, o) >= 32u)) {
            if (prof && lane == 0) atomicAdd(&S.cnt[CNT_PROF_SWITCHES], 1ull);
            // switch type: park the current particles on their stack
            if (S.ws[w].stk[t] + 32u > A.stack_cap) spill_to_queue(A, S, gw, w, t, 64u);
            const unsigned actm = __ballot_sync(FULL, p.act);
            const unsigned base = S.ws[w].stk[t];
            if (p.act) {
                const unsigned rank = __popc(actm & lanemask_lt());
                A.stacks[((size_t)gw * 2 + t) * A.stack_cap + base + rank] = make_rec(p);
                p.act = false;
            }
            __syncwarp();
            if (lane == 0) S.ws[w].stk[t] = base + __popc(actm);
            __syncwarp();
            t = o;
            continue;
        }
        if (prof) c0 = clock64();
        // headroom for this step's secondaries (at most two per lane)
        if (S.ws[w].stk[0] + 64u > A.stack_cap) spill_to_queue(A, S, gw, w, 0, 64u);
        if (S.ws[w].stk[1] + 64u > A.stack_cap) spill_to_queue(A, S, gw, w, 1, 64u);
        if (t == 0) {
            // Up to PH_FLIGHTS Woodcock flights per lane until its event is
            // real, then the real events' interactions together: with many
            // fictitious events (low densities under a high majorant) more
            // lanes reach an interaction per pass; in a homogeneous medium
            // every first flight is real and the loop ends at once.  The
            // energy, so its grid coordinate and majorant, stays the same
            // over the flights of a pass.
            uint32_t pidx = 0u, prz = 0u;
            bool real = false;
            const float xp = fmaf(__log2f((float)p.E), A.phys.grid.ph_a, A.phys.grid.ph_bq);
            const float mu_hat = p.act ? interp_ldg(S.plans[p.plan].maj, xp) : 1.0f;
            int rm = 0;
            float rrho = 0.f, rmu = 0.f;
            for (int k = 0; k < PH_FLIGHTS; ++k) {
                const bool fly = p.act && !real;
                const unsigned flym = __ballot_sync(FULL, fly);
                if (flym == 0u) break;
                if (fly) {
                    count(S, w, CNT_PH_EVENTS);
                    real = photon_flight<ONE>(A, S, p, xp, mu_hat, pidx, prz, rm, rrho, rmu, w);
                }
            }
            if (real) photon_interact<KERMA, ONE>(A, S, p, pidx, prz, xp, rm, rrho, rmu, gw, w);
        } else {
            // Up to EL_STEPS steps before the warp goes back to refill its
            // lanes, as long as three quarters of them are still stepping.  One
            // under the ablation's policies, which differ in the refill alone:
            // up to four there would make every fourth pass mean every 16th step
            // (every 16th pass of 1e6 electrons then takes 5.2 ms instead of 3.6).
            bool fin = p.act && p.E < A.phys.e_abs_q;
            if (fin) p.act = false;
            const int keep = n_act - n_act / 4;
#pragma unroll 1
            for (int k = 1;; ++k) {
                uint32_t dep_idx = 0, dep_e = 0;
                if (prof) {  // each step is a pass of its own in the profile
                    const unsigned stepm = __ballot_sync(FULL, p.act);
                    if (lane == 0) {
                        atomicAdd(&S.cnt[CNT_PROF_ITER + 1], 1ull);
                        atomicAdd(&S.cnt[CNT_PROF_LANES + 1], (unsigned long long)__popc(stepm));
                    }
                }
                if (p.act) {
                    count(S, w, CNT_E_STEPS);
                    electron_step<ONE>(A, S, p, gw, w, dep_idx, dep_e, fin);
                }
                const PlanDev &P = S.plans[p.plan];
                if (agg)
                    deposit_aggregated(P, p.hist, dep_idx, dep_e);
                else
                    deposit(P, p.hist, dep_idx, dep_e);
                const int alive = __popc(__ballot_sync(FULL, p.act));
                if (k == (SCHED ? 1 : EL_STEPS) || alive < keep || alive == 0) break;
            }
            if (fin) electron_end(S, p);
        }
        if (prof) {
            __syncwarp();
            if (lane == 0) {
                atomicAdd(&S.cnt[CNT_PROF_CYC + t], (unsigned long long)(clock64() - c0));
                if (t == 0) {
                    atomicAdd(&S.cnt[CNT_PROF_ITER], 1ull);
                    atomicAdd(&S.cnt[CNT_PROF_LANES], (unsigned long long)n_act);
                }
            }
        }
    }
    __syncthreads();
    for (int i = tid; i < CNT_N; i += blockDim.x) {
        unsigned long long n = cnt[i];
        if (row_word(i) < CNT_ROW)  // the cycle profile has no row
            for (int k = 0; k < MAX_WARPS; ++k) n += wcnt[k * CNT_ROW + row_word(i)];
        if (n) atomicAdd(&A.counters[i], n);
    }
    for (int i = tid; i < 3 * A.n_plans; i += blockDim.x)
        if (ledger[i]) atomicAdd(&plans[i / 3].ledger[i % 3], ledger[i]);
}

size_t transport_smem_bytes(uint32_t tab_bytes) { return (size_t)SMEM_FIXED + tab_bytes; }

// Instantiations by register budget.  A launch bound (threads, CTAs) caps the
// registers at 65536 / (threads x CTAs), and a kernel built for a budget runs
// any launch with no more threads per CTA and no more threads per SM than its
// bound: 128 registers up to 512 threads per SM, 80 up to 768, 64 up to 1024.
// The 64-register kernel is the production one at its default shape, 1024
// threads x 1 CTA per SM: the same 32 warps per SM as 512 x 2 but one copy of
// the tables in shared memory, which leaves the larger L1 carve-out to the
// voxel words, majorants and stack records (5-6% faster on the batched
// workload than 512 x 2 in a same-box A/B).  The profile, aggregation,
// refill-policy, photon-only and phase-space kernels are built for it too.
typedef void (*TransportKernel)(const TransportArgs);
// Launches of one plan have their own (ONE) for the production, photon-only and
// phase-space kernels.
struct Variant {
    int max_threads, min_blocks;
    bool prof, agg, sched, kerma, phsp, one;
    TransportKernel fn;
};
static const Variant kVariants[] = {
    {512, 1, false, false, false, false, false, false, k_transport<512, 1, false, false, false, false, false, false>},
    {384, 2, false, false, false, false, false, false, k_transport<384, 2, false, false, false, false, false, false>},
    {1024, 1, false, false, false, false, false, true, k_transport<1024, 1, false, false, false, false, false, true>},
    {1024, 1, false, false, false, false, false, false, k_transport<1024, 1, false, false, false, false, false, false>},
    {1024, 1, true, false, false, false, false, false, k_transport<1024, 1, true, false, false, false, false, false>},
    {1024, 1, false, true, false, false, false, false, k_transport<1024, 1, false, true, false, false, false, false>},
    {1024, 1, false, false, true, false, false, false, k_transport<1024, 1, false, false, true, false, false, false>},
    {1024, 1, false, false, false, true, false, true, k_transport<1024, 1, false, false, false, true, false, true>},
    {1024, 1, false, false, false, true, false, false, k_transport<1024, 1, false, false, false, true, false, false>},
    {1024, 1, false, false, false, false, true, true, k_transport<1024, 1, false, false, false, false, true, true>},
    {1024, 1, false, false, false, false, true, false, k_transport<1024, 1, false, false, false, false, true, false>},
};

// The first variant (most registers first) whose bound covers the launch.
static TransportKernel pick_variant(int block, int blocks_per_sm, bool prof, bool agg, bool sched, bool kerma,
                                    bool phsp, bool one) {
    for (const Variant &v : kVariants)
        if (v.prof == prof && v.agg == agg && v.sched == sched && v.kerma == kerma && v.phsp == phsp &&
            (one || !v.one) &&
            block <= v.max_threads && block * blocks_per_sm <= v.max_threads * v.min_blocks)
            return v.fn;
    return nullptr;
}

cudaError_t transport_configure() {
    for (const Variant &v : kVariants) {
        cudaError_t e = cudaFuncSetAttribute(v.fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)transport_smem_bytes(TAB_BYTES));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

const void *transport_kernel(const TransportArgs &a, int block, int blocks_per_sm) {
    return (const void *)pick_variant(block, blocks_per_sm, (a.flags & GPUMCD_LAUNCH_PROFILE) != 0u,
                                      (a.flags & GPUMCD_LAUNCH_WARP_AGGREGATE) != 0u, a.refill_period != 1u,
                                      (a.flags & GPUMCD_LAUNCH_KERMA) != 0u, a.phsp != 0u, a.n_plans == 1);
}

cudaError_t launch_transport(const TransportArgs &a, int grid, int block, int blocks_per_sm, cudaStream_t s) {
    TransportKernel fn = (TransportKernel)transport_kernel(a, block, blocks_per_sm);
    if (!fn) return cudaErrorInvalidConfiguration;
    if (a.tab_bytes < tab_bytes(1) || a.tab_bytes > (uint32_t)TAB_BYTES) return cudaErrorInvalidValue;
    fn<<<grid, block, transport_smem_bytes(a.tab_bytes), s>>>(a);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Energy grouping of a spectrum or a phase space (GPUMCD §IV): before a
// launch, a counting sort puts the plan's histories in decreasing order of
// their primary's energy bin, and the launch claims them in that order.  Each
// history starts as an ungrouped one does (the same draw, or the same record,
// in make_primary), so the tally does not change; warps, and the whole grid at
// any moment, start histories of similar energy, the longest first.
// ---------------------------------------------------------------------------
constexpr int GROUP_THREADS = 256;
// Histories a block sorts, in rounds of one a thread.  Each round waits for a
// key (a draw and a search, or a record), so a short sort wants many blocks; a
// long one wants fewer, as each adds its bins to the global counts.  Four
// rounds up to 2^19 histories, eight above, against sixteen throughout: the
// sort of 2e4 histories takes 23 us less, of 2e5 19, of 1e6 2, of 4e6 6.
static uint32_t group_per_block(uint32_t n) { return (n <= (1u << 19) ? 4u : 8u) * GROUP_THREADS; }

// Energy bins of a grouped phase space: 64 to an octave over [2^-10, 2^6) MeV,
// from the float's exponent and top six mantissa bits (exact and monotone for
// E > 0; energies outside the range share the end bins).
constexpr int PHSP_GROUP_BINS = GPUMCD_MAX_SPECTRUM_BINS;
static_assert(PHSP_GROUP_BINS == 1024, "16 octaves x 64 bins");

__device__ __forceinline__ int group_bins(const PlanDev &P) {
    return P.beam == GPUMCD_BEAM_PHASE_SPACE ? PHSP_GROUP_BINS : P.n_spec;
}

// The energy bin of history h's primary, counted from the top: a phase
// space's record h mod n, or the spectrum bin the history's own draw picks.
__device__ __forceinline__ int group_key(const PlanDev &P, unsigned long long h) {
    if (P.beam == GPUMCD_BEAM_PHASE_SPACE) {
        const float4 *ps = reinterpret_cast<const float4 *>(P.spec);
        const float E = __ldg(ps + 2 * (size_t)(h % (unsigned long long)P.n_phsp)).w;
        const int b = (int)(__float_as_uint(E) >> 17) - ((127 - 10) << 6);
        return PHSP_GROUP_BINS - 1 - min(max(b, 0), PHSP_GROUP_BINS - 1);
    }
    // draw 0 of the primary's lineage 1
    const uint4 r = philox4x32_10(make_uint4(0u, 1u, 0u, (uint32_t)h), make_uint2(P.key_lo, P.key_hi));
    return P.n_spec - 1 - spectrum_bin(P, u01(r.z));
}

// Count: each history's key, once, into keys[j]; the block's bin counts into
// count.  Lanes of a warp with the same key add once (one shared atomic per
// distinct key in the warp).
__global__ void __launch_bounds__(GROUP_THREADS) k_group_count(const __grid_constant__ PlanDev P, uint32_t n,
                                                               uint32_t per_block, unsigned *count,
                                                               uint16_t *keys) {
    __shared__ unsigned local[GPUMCD_MAX_SPECTRUM_BINS];
    const int nb = group_bins(P);
    const unsigned lt = lanemask_lt();
    // the block's histories in rounds of one per thread: the same trip count
    // for every thread, so whole warps take part in each match
    const uint32_t j0 = blockIdx.x * per_block, jend = min(n, j0 + per_block);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) local[i] = 0u;
    __syncthreads();
    for (uint32_t jb = j0; jb < jend; jb += blockDim.x) {
        const uint32_t j = jb + threadIdx.x;
        const int k = j < jend ? group_key(P, P.hist_base + j) : -1;
        const unsigned same = __match_any_sync(FULL, k);
        if (k >= 0) {
            keys[j] = (uint16_t)k;
            if ((same & lt) == 0u) atomicAdd(&local[k], (unsigned)__popc(same));
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += blockDim.x)
        if (local[i]) atomicAdd(&count[i], local[i]);
}

// Exclusive prefix sum of the bin counts, in place: one block of
// GPUMCD_MAX_SPECTRUM_BINS threads, a bin each (scans within the warps, then
// over the warps' totals).
constexpr int GROUP_SCAN_THREADS = GPUMCD_MAX_SPECTRUM_BINS;
__global__ void __launch_bounds__(GROUP_SCAN_THREADS) k_group_scan(unsigned *count, int n_bins) {
    __shared__ unsigned warp_sum[GROUP_SCAN_THREADS / 32];
    const int i = threadIdx.x, lane = i & 31, wid = i >> 5;
    const unsigned c = i < n_bins ? count[i] : 0u;
    unsigned v = c;  // inclusive scan within the warp
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const unsigned u = __shfl_up_sync(FULL, v, d);
        if (lane >= d) v += u;
    }
    if (lane == 31) warp_sum[wid] = v;
    __syncthreads();
    if (wid == 0) {
        unsigned t = lane < GROUP_SCAN_THREADS / 32 ? warp_sum[lane] : 0u;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const unsigned u = __shfl_up_sync(FULL, t, d);
            if (lane >= d) t += u;
        }
        if (lane < GROUP_SCAN_THREADS / 32) warp_sum[lane] = t;  // inclusive over the warps
    }
    __syncthreads();
    if (i < n_bins) count[i] = v - c + (wid > 0 ? warp_sum[wid - 1] : 0u);
}

// Each block reserves, per bin, room for its histories of that bin, then
// writes their offsets there (the order within a bin is not fixed: claims in
// any order give the same tally).  The keys come from k_group_count.
__global__ void __launch_bounds__(GROUP_THREADS) k_group_scatter(const __grid_constant__ PlanDev P, uint32_t n,
                                                                 uint32_t per_block, unsigned *cursor,
                                                                 const uint16_t *keys, uint32_t *order) {
    __shared__ unsigned local[GPUMCD_MAX_SPECTRUM_BINS];
    __shared__ unsigned base[GPUMCD_MAX_SPECTRUM_BINS];
    const int nb = group_bins(P);
    const int lane = threadIdx.x & 31;
    const unsigned lt = lanemask_lt();
    const uint32_t j0 = blockIdx.x * per_block, jend = min(n, j0 + per_block);
    for (int i = threadIdx.x; i < nb; i += blockDim.x) local[i] = 0u;
    __syncthreads();
    for (uint32_t jb = j0; jb < jend; jb += blockDim.x) {
        const uint32_t j = jb + threadIdx.x;
        const int k = j < jend ? (int)keys[j] : -1;
        const unsigned same = __match_any_sync(FULL, k);
        if (k >= 0 && (same & lt) == 0u) atomicAdd(&local[k], (unsigned)__popc(same));
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nb; i += blockDim.x) {
        base[i] = local[i] ? atomicAdd(&cursor[i], local[i]) : 0u;
        local[i] = 0u;
    }
    __syncthreads();
    for (uint32_t jb = j0; jb < jend; jb += blockDim.x) {
        const uint32_t j = jb + threadIdx.x;
        const int k = j < jend ? (int)keys[j] : -1;
        const unsigned same = __match_any_sync(FULL, k);
        const int leader = __ffs(same) - 1;
        unsigned slot = 0u;
        if (k >= 0 && lane == leader) slot = atomicAdd(&local[k], (unsigned)__popc(same));
        slot = __shfl_sync(FULL, slot, leader);
        if (k >= 0) order[base[k] + slot + (unsigned)__popc(same & lt)] = j;
    }
}

cudaError_t launch_group_order(const PlanDev &P, uint32_t n, unsigned *count, uint16_t *keys, uint32_t *order,
                               cudaStream_t s) {
    const int nb = P.beam == GPUMCD_BEAM_PHASE_SPACE ? (P.n_phsp > 0 ? PHSP_GROUP_BINS : 0) : P.n_spec;
    if (nb < 1 || nb > GPUMCD_MAX_SPECTRUM_BINS || n == 0 || !P.spec) return cudaErrorInvalidValue;
    cudaError_t e = cudaMemsetAsync(count, 0, (size_t)nb * sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    const uint32_t per_block = group_per_block(n);
    const unsigned blocks = (n + per_block - 1) / per_block;
    k_group_count<<<blocks, GROUP_THREADS, 0, s>>>(P, n, per_block, count, keys);
    k_group_scan<<<1, GROUP_SCAN_THREADS, 0, s>>>(count, nb);
    k_group_scatter<<<blocks, GROUP_THREADS, 0, s>>>(P, n, per_block, count, keys, order);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Sampler diagnostics: the same device samplers, one draw per thread.
// ---------------------------------------------------------------------------
__global__ void k_debug_sample(const float *tabg, Phys ph, int kind, float p0, int material,
                               const float *spec, int n_spec, uint64_t n, uint64_t seed, float *out) {
    const uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    PlanDev P{};
    const uint2 k = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    const auto key = [k](int r) { return philox_round_key(k, r); };
    P.spec = spec;
    P.n_spec = n_spec;
    Lane p;
    p.hist = (uint32_t)i;
    p.lin = philox_lineage((uint32_t)(i >> 32), 0x5EEDu, key(0), key(1));
    p.draw = 0;
    p.plan = 0;
    float v = 0.f;
    uint32_t wd;
    unsigned capped = 0;
    if (kind == 0 || kind == 6) {
        float c;
        const float eps = sample_kn(p, key, p0 / kMC2f, &c, &wd, &capped);
        v = kind == 0 ? c : eps;
    } else if (kind == 1) {
        v = sample_sauter(p, key, p0, &wd, &capped);
    } else if (kind == 2) {
        v = sample_hard(p, key, true, p0, ph.t_c, 0.f, 0.f, &wd, &capped);
    } else if (kind == 3) {
        v = sample_hard(p, key, false, p0, ph.k_c, __ldg(tabg + TAB_BREM + 2 * material),
                        __ldg(tabg + TAB_BREM + 2 * material + 1), &wd, &capped);
    } else if (kind == 4) {
        // the transport's own ms_mu, given the tables in global memory instead
        // of their shared-memory copy (the same word of the draw as a step uses)
        const uint4 r = draw4(p, key);
        v = ms_mu(tabg, ph.grid, p0, u01(r.z));
    } else if (kind == 5) {
        const uint4 r = draw4(p, key);
        v = sample_spectrum(P, u01(r.z));
    }
    out[i] = capped ? __int_as_float(0x7fc00000) : v;  // a capped draw shows up as NaN
}

cudaError_t launch_debug_sample(const float *tab, const Phys &phys, int kind, float p0, int material,
                                const float *spec, int n_spec, uint64_t n, uint64_t seed, float *out,
                                cudaStream_t s) {
    const int grid = (int)((n + 255) / 256);
    k_debug_sample<<<grid ? grid : 1, 256, 0, s>>>(tab, phys, kind, p0, material, spec, n_spec, n, seed, out);
    return cudaGetLastError();
}

}  // namespace gm
