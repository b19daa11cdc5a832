// ocmc_transport.cu -- persistent coupled photon-electron transport kernel.
//
// Method (Tian et al., Sec. 2.1): photons fly by Woodcock tracking against a
// phantom-wide majorant and interact by Compton scattering, photoelectric
// absorption or pair production; electrons and positrons take Class II
// condensed-history steps d = min(d_vox, d_maxs, d_maxe, d_event), each inside
// one voxel, with a random-hinge multiple-scattering deflection, CSDA energy
// loss deposited in the step's voxel, and discrete Moller / bremsstrahlung
// events sampled by Woodcock tracking in energy; positrons annihilate into two
// photons at the end of their track.
//
// Scheduling (Sec. 2.2.1, Table 1): the paper launches batches of up to M
// particles of one type, taken from the photon stack, the electron stack or
// the source. Here every warp runs that loop by itself inside one persistent
// launch: its 32 lanes always hold particles of one kind (warp mode: photons,
// or charged particles, which wait on two stacks split by energy class); once
// enough lanes are free they refill from the warp's own stack of that kind,
// then from the source (energy-sorted history ids from a global counter); the
// warp moves to the fullest other stack when its lanes run dry or that stack
// grows large. Secondaries are pushed to the warp's stacks. A warp ends when
// the source is exhausted and its stacks are empty; no warp ever waits on
// another.
//
// What bounds it: instruction issue and instruction fetch, not memory (DRAM 2 % of its rate). A warp
// instruction carries about 19 of 32 lanes because steps differ, and the kernel is larger than an
// SM's instruction caches, so the code is kept small and uniform: one copy of everything that ends or
// emits a particle (finish), 32-bit event counters (a 64-bit shared add is a loop per lane), the first
// draws of a step taken straight from its random block, geometric crossings and post-hinge crossings
// through one piece of code, no branches in the face distances and the rotation, and a scheduler that
// is skipped while no lane and no stack needs it. 1e8 6 MV photons on the 120^3 slab take 96 ms, 1e7
// electrons of 15 MeV on the half-slab 62.7; one copy of each kind of code, the refill thresholds
// (REFILL_G), the held events (HELD) and k_chains each say below what they gave of that.
//
// Dose tally (Sec. 2.2.2): 64-bit fixed-point integer atomics (2^-28 MeV
// units) into the tally of batch (history id mod B). Integer addition is
// associative and every particle's random stream is keyed by its lineage, so
// the tally is bit-identical for any launch configuration and timing.
#include "ocmc_device.cuh"

#include <algorithm>

namespace ocmc {

namespace {

constexpr unsigned FULL = 0xFFFFFFFFu;
constexpr int MAX_WARPS = 32;
constexpr int STEP_LIMIT = 1 << 22;
constexpr int HELD_MIN = 6;
constexpr int CHAIN_LANES = 8;    // a warp flies chains together while at most this many photons are left in it
constexpr int CHAIN_STEPS = 24;   // flights in a row that make a chain (a photon makes about 6 in water)
constexpr uint32_t CHAIN_MAX_N = 4u * STEP_LIMIT;   // draws after which a photon is left to its steps and their limit

// Block statistics in shared memory: event counts as 32-bit words (shared memory adds 32-bit
// integers natively and a warp's lanes together; a 64-bit shared add is a compare-and-swap loop
// per lane), the energy sums that hot paths add to as 32-bit halves. Counts move to the
// 64-bit totals in global memory before a word can wrap (flush_stats) and when a warp ends.
struct BlockStats {
    unsigned int n[ST_E_IN];       // event counts, slots [0, ST_E_IN)
    unsigned int e[3][2];          // energy sums ST_E_IN .. ST_E_MISS: low and high words
};
enum { BE_IN = 0, BE_ESC, BE_MISS };
static_assert(ST_E_ESC - ST_E_IN == BE_ESC && ST_E_MISS - ST_E_IN == BE_MISS, "the block's sums in the totals' order");

// Source and tally of a launch, compile-time so that each kernel carries only its own code: one beam
// with a dense tally per statistical batch, beamlets with a dense tally each (a particle's batch is
// then its beamlet), or beamlets with sparse hash tallies.
enum { ONE_BEAM = 0, BEAMLETS_DENSE, BEAMLETS_HASH };

template <int BL>
struct CtxT {
    static constexpr bool beamlets = BL != ONE_BEAM, hashed = BL == BEAMLETS_HASH;
    const TransportArgs& a;
    const SmemTables& T;
    PRec* stk;                   // warp's stacks: [0, cap) photons, [cap, 2cap) charged, [2cap, 3cap) slow charged
    int* top;                    // shared: top[0] photons, top[1] charged, top[2] charged below e_split
    BlockStats* st;              // shared block statistics
    float inv_dx, inv_dy, inv_dz, Lx, Ly, Lz;
};

// one event of kind k
template <class C>
__device__ __forceinline__ void count(C& c, int k) { atomicAdd(&c.st->n[k], 1u); }

// what hardly ever happens goes straight to the totals (not the energy of particles that miss the phantom:
// 1.6e7 photons, two thirds of which miss, took 10.6 ms with a global atomic each, 3.5 without)
template <class C>
__device__ __forceinline__ void count_rare(C& c, int k, unsigned long long v) { atomicAdd(c.a.stats + k, v); }

template <class C>
__device__ __forceinline__ void add_energy(C& c, int k, unsigned long long q)
{
    const unsigned lo = (unsigned)q, hi = (unsigned)(q >> 32);
    const unsigned old = atomicAdd(&c.st->e[k][0], lo);
    const unsigned carry = hi + (old > ~lo ? 1u : 0u);
    if (carry) atomicAdd(&c.st->e[k][1], carry);
}

// Checks build: a lane whose voxel index lies outside the grid flags ERR_BOUNDS (and its
// particle is ended by the caller before any access). Always false in the normal build.
template <class C>
__device__ __forceinline__ bool vox_bad(const C& c, const Lane& p)
{
    if constexpr (OCMC_CHECKS) {
        if (p.ix < 0 || p.iy < 0 || p.iz < 0 || p.ix >= c.a.nx || p.iy >= c.a.ny || p.iz >= c.a.nz) {
            atomicOr(c.a.err, ERR_BOUNDS);
            return true;
        }
    }
    return false;
}

// Stack of a waiting charged particle: 1, or 2 below the energy-class boundary (e_split is 0
// when the warps keep a single charged stack, so that everything then goes to stack 1).
__device__ __forceinline__ int charged_stack(const TransportArgs& a, float E) { return E < a.e_split ? 2 : 1; }

// fixed-point energy (round to nearest even) with 32-bit conversions only: below 2^32 units
// (16 MeV) directly; above, q is a float >= 2^32 and therefore a multiple of 2^9, so q / 2^8 is
// an integer below 2^32 for any energy under 4 GeV and the result is exact (no 64-bit
// float-to-integer conversion, which would occupy the FP64 pipe)
__device__ __forceinline__ unsigned long long fx(float e)
{
    float q = e * TALLY_SCALE;
    return q < 4294967040.f ? (unsigned long long)__float2uint_rn(q)
                            : (unsigned long long)__float2uint_rn(q * 0.00390625f) << 8;
}

// Batched-beamlet tally: add q to voxel v of beamlet b's open-addressing table
// (linear probing, key claimed by compare-and-swap). A full table sets the
// beamlet's overflow flag; the host then enlarges that table and runs again.
__device__ __forceinline__ void hash_add(const TransportArgs& a, uint32_t b, uint32_t v, unsigned long long q)
{
    const BeamletDev& B = a.beamlets[b];
    unsigned int* keys = a.bl_keys + B.table_off;
    unsigned long long* vals = a.bl_vals + B.table_off;
    const uint32_t mask = B.cap_mask;
    uint32_t h = v * 0x9E3779B1u;
    uint32_t s = (h ^ (h >> 15)) & mask;
    for (int probe = 0; probe <= (int)min(mask, 4095u); ++probe) {
        uint32_t k = *((volatile unsigned int*)(keys + s));
        if (k == BL_EMPTY) k = atomicCAS(keys + s, BL_EMPTY, v);
        if (k == BL_EMPTY || k == v) {
            atomicAdd(vals + s, q);
            return;
        }
        s = (s + 1u) & mask;
    }
    atomicOr(a.bl_overflow + b, 1u);
}

// add q fixed-point units to the lane's tally at voxel (ix, iy, iz)
template <class C>
__device__ __forceinline__ void deposit_q(C& c, const Lane& p, int ix, int iy, int iz, unsigned long long q)
{
    if (q) {
        const int v = ix + c.a.nx * (iy + c.a.ny * iz);     // grids have at most 1024^3 voxels
        if constexpr (OCMC_CHECKS) {
            if (ix < 0 || iy < 0 || iz < 0 || ix >= c.a.nx || iy >= c.a.ny || iz >= c.a.nz ||
                (!C::beamlets && (p.batch < 0 || p.batch >= c.a.pp.n_batches)) ||
                (C::beamlets && !C::hashed && (p.batch < 0 || p.batch >= c.a.n_beamlets))) {
                atomicOr(c.a.err, ERR_BOUNDS);
                return;
            }
        }
        if constexpr (C::hashed) hash_add(c.a, p.r.h1 & ~BL_TAG, (uint32_t)v, q);
        else atomicAdd(c.a.tally + (long long)p.batch * c.a.nvox + v, q);
    }
}

// energy dE > 0 (nothing otherwise) to voxel (ix, iy, iz)
template <class C>
__device__ __forceinline__ void deposit(C& c, const Lane& p, int ix, int iy, int iz, float dE)
{
    deposit_q(c, p, ix, iy, iz, dE > 0.f ? fx(dE) : 0ull);
}

// a particle at p's position on stack t
template <class C>
__device__ __forceinline__ void push(C& c, int t, const Lane& p, float E, float u, float v, float w, int type, uint32_t sub,
                                     uint32_t n)
{
    int slot = atomicAdd(c.top + t, 1);
    if (slot >= c.a.cap) {
        atomicOr(c.a.err, ERR_OVERFLOW);
        count_rare(c, ST_DROPPED, 1);
        count_rare(c, ST_E_DROPPED, fx(E));
        return;
    }
    uint32_t vt = (uint32_t)p.ix | ((uint32_t)p.iy << 10) | ((uint32_t)p.iz << 20) | ((uint32_t)type << 30);
    uint4* q = reinterpret_cast<uint4*>(c.stk + (size_t)t * c.a.cap + slot);
    q[0] = make_uint4(__float_as_uint(p.x), __float_as_uint(p.y), __float_as_uint(p.z), __float_as_uint(E));
    q[1] = make_uint4(__float_as_uint(u), __float_as_uint(v), __float_as_uint(w), vt);
    q[2] = make_uint4(p.r.h0, p.r.h1, sub, n);
}

template <class C>
__device__ __forceinline__ void pop_lane(const C& c, int t, int slot, Lane& p)
{
    if constexpr (OCMC_CHECKS) {
        if (slot < 0 || slot >= c.a.cap || t < 0 || t >= c.a.nstk) {
            atomicOr(c.a.err, ERR_BOUNDS);
            slot = 0;
            t = 0;
        }
    }
    const uint4* q = reinterpret_cast<const uint4*>(c.stk + (size_t)t * c.a.cap + slot);
    uint4 a = q[0], b = q[1], d = q[2];
    p.x = __uint_as_float(a.x); p.y = __uint_as_float(a.y); p.z = __uint_as_float(a.z); p.E = __uint_as_float(a.w);
    p.u = __uint_as_float(b.x); p.v = __uint_as_float(b.y); p.w = __uint_as_float(b.z);
    p.ix = b.w & 1023u; p.iy = (b.w >> 10) & 1023u; p.iz = (b.w >> 20) & 1023u; p.type = b.w >> 30;
    p.r.h0 = d.x; p.r.h1 = d.y; p.r.sub = d.z; p.r.n = d.w;
    if constexpr (C::beamlets) p.batch = (int)(d.y & ~BL_TAG);
    else p.batch = batch_of(d.x, d.y ^ c.a.stream_tag, c.a.pp.n_batches);
    p.steps = 0;
}

// What a step leaves to the loop's common tail (finish): the lane's fate and at most one secondary
// at the lane's position. One copy of the code that pushes, absorbs, annihilates and counts escapes
// serves every kind of step: with a copy at each place that ends or emits a particle the kernel was
// 88 KB of instructions and waited for instruction fetches more than for anything else.
enum { LIVE = 0, GONE, ESCAPED, ABSORBED, MOVED };   // MOVED: to the stack of its kind
struct Pend {
    float E, u, v, w;
    int type;                    // -1: no secondary
    uint32_t sub;
};

// Pair production: e- and e+ along the photon, sharing E - 2 mc^2 uniformly: the e- is the step's
// secondary, the lane itself becomes the e+.
template <class C>
__device__ __forceinline__ int pair_event(C& c, Lane& p, Pend& s)
{
    count(c, ST_PAIR);
    float avail = p.E - 2.f * MC2F;
    float Tm = rng_u(p.r, c.a.key0, c.a.key1) * avail, Tp = avail - Tm;
    s.E = Tm; s.u = p.u; s.v = p.v; s.w = p.w;
    s.type = ELECTRON;
    s.sub = child_sub(p.r.sub, p.r.n, 0);
    p.r.sub = child_sub(p.r.sub, p.r.n, 1);
    p.r.n = 0;
    p.E = Tp;
    p.type = POSITRON;
    return Tp >= c.a.pp.e_abs_e && !(c.a.pp.flags & 8) ? MOVED : ABSORBED;
}

// One Woodcock flight and, if real, the interaction.
template <class C>
__device__ __forceinline__ int photon_step(C& c, Lane& p, Pend& sec)
{
    const TransportArgs& a = c.a;
    const SmemTables& T = c.T;
    const uint32_t k0 = a.key0, k1 = a.key1;
    rng_step_start(p.r, k0, k1);
    EIdx ei = e_index(p.E);
    float lnmaj = lerp1(T.phmaj[ei.i], T.phmaj[ei.i + 1], ei.f);
    if (lnmaj < -1e29f) return ESCAPED;
    float mumax = __expf(lnmaj);
    float s = -__logf(u01(p.r.buf.x)) / mumax;         // the step's first three draws
    const float u_real = u01(p.r.buf.y), xi = u01(p.r.buf.z);
    p.x = fmaf(s, p.u, p.x);
    p.y = fmaf(s, p.v, p.y);
    p.z = fmaf(s, p.w, p.z);
    if (!(p.x >= 0.f && p.y >= 0.f && p.z >= 0.f && p.x <= c.Lx && p.y <= c.Ly && p.z <= c.Lz)) {
        if ((a.pp.flags & 4) && p.z > c.Lz) {
            count_rare(c, ST_TRANSMITTED, 1);
            count_rare(c, ST_E_TRANS, fx(p.E));
        }
        return ESCAPED;
    }
    p.ix = min((int)(p.x * c.inv_dx), a.nx - 1);
    p.iy = min((int)(p.y * c.inv_dy), a.ny - 1);
    p.iz = min((int)(p.z * c.inv_dz), a.nz - 1);
    const int vox = p.ix + a.nx * (p.iy + a.ny * p.iz);
    float rho = __ldg(a.density + vox);
    int m = __ldg(a.material + vox);
    float4 pa = T.ph[m * MS4 + ei.i], pb = T.ph[m * MS4 + ei.i + 1];
    float mu = rho * __expf(lerp1(pa.x, pb.x, ei.f));
    if (mu > mumax * 1.00001f) count_rare(c, ST_VIOL, 1);
    p.r.n += 2u;
    if (u_real * mumax >= mu) { count(c, ST_FICT); return LIVE; }
    if (a.pp.flags & 4) { count_rare(c, ST_E_KILLED, fx(p.E)); return GONE; }
    float fC = lerp1(pa.y, pb.y, ei.f), fP = lerp1(pa.z, pb.z, ei.f);
    p.r.n += 1u;
    if (xi >= fC && xi < fC + fP) {
        count(c, ST_PHOTO);
        return ABSORBED;
    }
    if (xi >= fC + fP && p.E > 2.f * MC2F) return pair_event(c, p, sec);
    // Compton scattering (also the rare pair selection below threshold from table interpolation)
    count(c, ST_COMPTON);
    float eps;
    bool ok = true;
    float cth = sample_compton(p.E, p.r, k0, k1, &eps, &ok);
    if (!ok) atomicOr(a.err, ERR_LIMIT);
    float xphi = rng_u(p.r, k0, k1);
    float E0 = p.E, E1 = __fmul_rn(eps, E0), Te = __fsub_rn(E0, E1);
    float u0 = p.u, v0 = p.v, w0 = p.w;
    rotate(p.u, p.v, p.w, cth, xphi);
    if (Te > 0.f) {
        float qu = __fsub_rn(__fmul_rn(E0, u0), __fmul_rn(E1, p.u)), qv = __fsub_rn(__fmul_rn(E0, v0), __fmul_rn(E1, p.v)),
              qw = __fsub_rn(__fmul_rn(E0, w0), __fmul_rn(E1, p.w));
        float inv = rsqrtf(fmaxf(__fmaf_rn(qw, qw, __fmaf_rn(qu, qu, __fmul_rn(qv, qv))), 1e-30f));
        sec.E = Te; sec.u = qu * inv; sec.v = qv * inv; sec.w = qw * inv;
        sec.type = ELECTRON;
        sec.sub = child_sub(p.r.sub, p.r.n, 0);
    }
    p.E = E1;
    return p.E < a.pp.e_abs_g ? ABSORBED : LIVE;
}

// the neighbouring voxel across a face, the position put exactly on it; false outside the phantom
template <class C>
__device__ __forceinline__ bool cross_face(const C& c, Lane& p, int face)
{
    const int ax = face >> 1, up = face & 1;
    const int i = (ax == 0 ? p.ix : ax == 1 ? p.iy : p.iz) + 2 * up - 1;
    const float x = (float)(i + 1 - up) * (ax == 0 ? c.a.dx : ax == 1 ? c.a.dy : c.a.dz);
    const int n = ax == 0 ? c.a.nx : ax == 1 ? c.a.ny : c.a.nz;
    if (ax == 0) { p.ix = i; p.x = x; }
    if (ax == 1) { p.iy = i; p.y = x; }
    if (ax == 2) { p.iz = i; p.z = x; }
    return (unsigned)i < (unsigned)n;
}

// Discrete hard event at the end of a step: Moller (probability sM / tot) or bremsstrahlung.
template <class C>
__device__ __forceinline__ void hard_event(C& c, Lane& p, int m, float sM, float tot, Pend& sec)
{
    const SmemTables& T = c.T;
    const float Tk = p.E;
    const bool moller = rng_u(p.r, c.a.key0, c.a.key1) * tot < sM;
    bool ok = true;
    float mu, W, mu1 = 1.f;
    if (moller) {
        count(c, ST_MOLLER);
        float eps = sample_moller(Tk, c.a.pp.w_cc, p.r, c.a.key0, c.a.key1, &ok);
        W = eps * Tk;
        float T1 = Tk - W;
        mu1 = sqrtf(fminf(1.f, T1 * (Tk + 2.f * MC2F) / (Tk * (T1 + 2.f * MC2F))));
        mu = sqrtf(fminf(1.f, W * (Tk + 2.f * MC2F) / (Tk * (W + 2.f * MC2F))));
    } else {
        count(c, ST_BREMS);
        W = sample_brems(Tk, c.a.pp.w_cb, T.msc[m * MS1], T.msc[m * MS1 + 1], p.r, c.a.key0, c.a.key1, &ok);
        float th = MC2F / (Tk + MC2F);
        mu = __cosf(th);
    }
    if (!ok) atomicOr(c.a.err, ERR_LIMIT);
    float xphi = rng_u(p.r, c.a.key0, c.a.key1);
    sec.E = W;
    sec.u = p.u; sec.v = p.v; sec.w = p.w;
    rotate(sec.u, sec.v, sec.w, mu, moller ? xphi + 0.5f : xphi);
    sec.type = moller ? ELECTRON : PHOTON;
    sec.sub = child_sub(p.r.sub, p.r.n, moller ? 2u : 3u);
    if (moller) rotate(p.u, p.v, p.w, mu1, xphi);      // a bremsstrahlung electron keeps its direction
    p.E = Tk - W;
}

// The candidate hard event of a lane that has waited with it: what charged_step does otherwise at the end
// of the step, with the material and the random block fetched again. (Written out in both places: with one
// function for both, the kernel without waiting ran 0.3 % slower.)
template <class C>
__device__ __forceinline__ int held_candidate(C& c, Lane& p, float sighat, Pend& sec)
{
    const TransportArgs& a = c.a;
    const SmemTables& T = c.T;
    if (vox_bad(c, p)) return GONE;
    const int m = __ldg(a.material + (p.ix + a.nx * (p.iy + a.ny * p.iz))), mb = m * MS4;
    if (p.r.n & 3u) p.r.buf = philox_block(p.r.n >> 2, p.r.h0, p.r.h1, p.r.sub, a.key0, a.key1);
    EIdx e2 = e_index(p.E);
    float4 A2 = T.el[mb + e2.i], B2 = T.el[mb + e2.i + 1];
    float sM = p.E > 2.f * a.pp.w_cc ? lerp1(A2.z, B2.z, e2.f) : 0.f;
    float sB = p.E > a.pp.w_cb ? lerp1(A2.w, B2.w, e2.f) : 0.f;
    float tot = sM + sB;
    if (tot > sighat * 1.00001f) count_rare(c, ST_VIOL, 1);
    if (rng_u(p.r, a.key0, a.key1) * sighat < tot) {
        hard_event(c, p, m, sM, tot, sec);
        if (p.E < a.pp.e_abs_e) return ABSORBED;
    } else {
        count(c, ST_HARD_FICT);
    }
    return LIVE;
}

// One condensed-history step. With HELD a candidate hard event at its end is left to held_candidate, and
// *held receives its majorant.
template <bool HELD, class C>
__device__ __forceinline__ int charged_step(C& c, Lane& p, Pend& sec, float* held)
{
    const TransportArgs& a = c.a;
    const SmemTables& T = c.T;
    const uint32_t k0 = a.key0, k1 = a.key1;
    if (vox_bad(c, p)) return GONE;
    const int vox = p.ix + a.nx * (p.iy + a.ny * p.iz);
    float rho = __ldg(a.density + vox);
    int m = __ldg(a.material + vox);
    int face;
    float sv = dist_to_face(p.x, p.y, p.z, p.u, p.v, p.w, p.ix, p.iy, p.iz, a.dx, a.dy, a.dz, &face);
    const int mb = m * MS4, mb2 = m * MS2;
    float hx = p.x, hy = p.y, hz = p.z, l2 = sv, sighat = 0.f;
    int lim = 0;
    bool crossed = true;
    // nothing to interact with, or a boundary closer than s_min: cross geometrically
    const bool geo = !(rho > 0.f) || sv < a.pp.s_min;
    if (geo) {
        count(c, ST_GEO);
    } else {
        rng_step_start(p.r, k0, k1);
        EIdx ei = e_index(p.E);
        float4 A = T.el[mb + ei.i], B = T.el[mb + ei.i + 1];
        float2 C2 = T.el2[mb2 + ei.i], D2 = T.el2[mb2 + ei.i + 1];
        float lnR = lerp1(A.x, B.x, ei.f);
        float s_maxe = lerp1(C2.x, D2.x, ei.f) / rho;
        sighat = (a.pp.flags & 1) ? 0.f : C2.y;
        // the step's draws in order: event distance (only with a majorant), hinge, deflection, azimuth
        const bool ev = sighat > 0.f;
        const uint32_t w1 = ev ? p.r.buf.y : p.r.buf.x, w2 = ev ? p.r.buf.z : p.r.buf.y, w3 = ev ? p.r.buf.w : p.r.buf.z;
        float d_ev = ev ? -__logf(u01(p.r.buf.x)) / (rho * sighat) : 3.0e38f;
        p.r.n += ev ? 2u : 1u;
        float s = sv;
        if (a.pp.d_maxs < s) { s = a.pp.d_maxs; lim = 1; }
        if (s_maxe < s) { s = s_maxe; lim = 2; }
        if (d_ev < s) { s = d_ev; lim = 3; }
        // random hinge: s1 straight, deflect, then the rest (clipped to this voxel)
        float s1 = u01(w1) * s;
        hx = fmaf(s1, p.u, p.x);
        hy = fmaf(s1, p.v, p.y);
        hz = fmaf(s1, p.w, p.z);
        float E0 = p.E;
        const float R0 = __expf(lnR), g0 = range_to_lnE(T, m, lnR);
        float Eend = csda_end2(T, m, E0, R0, g0, rho * s);
        if (!(a.pp.flags & 2)) {
            EIdx em = e_index(0.5f * (E0 + Eend));
            float l1 = lerp1(T.el[mb + em.i].y, T.el[mb + em.i + 1].y, em.f);
            const float G1 = rho * s * l1;
            const bool deflects = G1 >= 1e-12f;
            float cth = sample_ms_u(T, G1, u01(w2));
            p.r.n += deflects ? 2u : 1u;
            rotate(p.u, p.v, p.w, cth, u01(deflects ? w3 : w2));
        }
        float tex = dist_to_face(hx, hy, hz, p.u, p.v, p.w, p.ix, p.iy, p.iz, a.dx, a.dy, a.dz, &face);
        const float rem = s - s1;
        crossed = !(rem < tex);
        l2 = crossed ? tex : rem;
        if (crossed) Eend = csda_end2(T, m, E0, R0, g0, rho * (s1 + tex));
        deposit(c, p, p.ix, p.iy, p.iz, E0 - Eend);
        p.E = Eend;
    }
    p.x = fmaf(l2, p.u, hx);
    p.y = fmaf(l2, p.v, hy);
    p.z = fmaf(l2, p.w, hz);
    if (crossed && !cross_face(c, p, face)) return ESCAPED;
    if (geo) return LIVE;
    if (p.E < a.pp.e_abs_e) return ABSORBED;
    if (lim == 3 && !crossed) {
        if constexpr (HELD) {
            *held = sighat;
            return LIVE;
        }
        EIdx e2 = e_index(p.E);
        float4 A2 = T.el[mb + e2.i], B2 = T.el[mb + e2.i + 1];
        float sM = p.E > 2.f * a.pp.w_cc ? lerp1(A2.z, B2.z, e2.f) : 0.f;
        float sB = p.E > a.pp.w_cb ? lerp1(A2.w, B2.w, e2.f) : 0.f;
        float tot = sM + sB;
        if (tot > sighat * 1.00001f) count_rare(c, ST_VIOL, 1);
        if (rng_u(p.r, k0, k1) * sighat < tot) {
            hard_event(c, p, m, sM, tot, sec);
            if (p.E < a.pp.e_abs_e) return ABSORBED;
        } else {
            count(c, ST_HARD_FICT);
        }
    }
    return LIVE;
}

// ---- voxel-crossing (fixed-step) electron steps ------------------------------------------
// The stepping scheme the paper contrasts with its own (Sec. 4): a step is not stopped at voxel
// faces. s = min(d_maxs, d_maxe, d_event) with d_maxe from the step's first voxel and d_event
// sampled against the phantom-wide majorant of rho * sigma_hard (so a candidate may fall in any
// voxel); random hinge at xi s with the multiple-scattering angle of the whole step in the first
// voxel's medium; along both straight parts the CSDA loss of each traversed voxel's own
// material and density is deposited there; the step ends early where the energy reaches
// E (1 - f_maxe) (before the hinge: deflected there, for the path travelled); a candidate at the
// end of an event-limited step is real with probability rho sigma_hard(E) / majorant in the
// voxel where it ends.
enum { SEG_DONE = 0, SEG_FLOOR, SEG_OUT, SEG_ABSORBED, SEG_GONE };

__device__ __forceinline__ float range_R(const SmemTables& T, int m, float E)
{
    const EIdx ei = e_index(E);
    return __expf(lerp1(T.el[m * MS4 + ei.i].x, T.el[m * MS4 + ei.i + 1].x, ei.f));
}

// Moves p a path length L along its direction through the voxels, losing and depositing the
// CSDA energy of each voxel it crosses; stops early at the energy floor Ef, on absorption or on
// escape. *done receives the path length travelled.
template <class C>
__device__ __forceinline__ int cross_segment(C& c, Lane& p, float L, float Ef, float* done)
{
    const TransportArgs& a = c.a;
    const SmemTables& T = c.T;
    float left = L, moved = 0.f;
    int r = SEG_DONE;
    for (int guard = 0; left > 0.f && r == SEG_DONE; ++guard) {
        if (guard > 4 * (a.nx + a.ny + a.nz)) { atomicOr(a.err, ERR_LIMIT); break; }   // cannot happen: bounded crossings
        if (vox_bad(c, p)) { r = SEG_GONE; break; }
        const int vox = p.ix + a.nx * (p.iy + a.ny * p.iz);
        const float rho = __ldg(a.density + vox);
        const int m = __ldg(a.material + vox);
        int face;
        const float sv = dist_to_face(p.x, p.y, p.z, p.u, p.v, p.w, p.ix, p.iy, p.iz, a.dx, a.dy, a.dz, &face);
        float l = left, Eend = p.E;
        bool cross = false, flo = false;
        if (sv < l) { l = sv; cross = true; }
        if (rho > 0.f) {
            const EIdx ei = e_index(p.E);
            const float lnR = lerp1(T.el[m * MS4 + ei.i].x, T.el[m * MS4 + ei.i + 1].x, ei.f);
            const float R = __expf(lnR);
            const float lf = (R - range_R(T, m, Ef)) / rho;
            if (lf <= l) { l = fmaxf(lf, 0.f); cross = false; flo = true; Eend = Ef; }
            else Eend = csda_end2(T, m, p.E, R, range_to_lnE(T, m, lnR), rho * l);
        }
        p.x = fmaf(l, p.u, p.x);
        p.y = fmaf(l, p.v, p.y);
        p.z = fmaf(l, p.w, p.z);
        deposit(c, p, p.ix, p.iy, p.iz, p.E - Eend);
        p.E = Eend;
        left -= l;
        moved += l;
        if (p.E < a.pp.e_abs_e) r = SEG_ABSORBED;
        else if (flo) r = SEG_FLOOR;
        else if (cross && !cross_face(c, p, face)) r = SEG_OUT;
    }
    *done = moved;
    return r;
}

__device__ __forceinline__ int segment_fate(int r) { return r == SEG_OUT ? ESCAPED : r == SEG_ABSORBED ? ABSORBED : GONE; }

template <class C>
__device__ __forceinline__ int charged_step_cross(C& c, Lane& p, Pend& sec)
{
    const TransportArgs& a = c.a;
    const SmemTables& T = c.T;
    const uint32_t k0 = a.key0, k1 = a.key1;
    if (vox_bad(c, p)) return GONE;
    const int vox = p.ix + a.nx * (p.iy + a.ny * p.iz);
    const float rho0 = __ldg(a.density + vox);
    const int m0 = __ldg(a.material + vox);
    if (!(rho0 > 0.f)) {                       // no matter here: fly to the next voxel
        int face;
        float sv = dist_to_face(p.x, p.y, p.z, p.u, p.v, p.w, p.ix, p.iy, p.iz, a.dx, a.dy, a.dz, &face);
        p.x = fmaf(sv, p.u, p.x);
        p.y = fmaf(sv, p.v, p.y);
        p.z = fmaf(sv, p.w, p.z);
        count(c, ST_GEO);
        return cross_face(c, p, face) ? LIVE : ESCAPED;
    }
    rng_step_start(p.r, k0, k1);
    const float E0 = p.E;
    const EIdx ei = e_index(E0);
    const int mb = m0 * MS4, mb2 = m0 * MS2;
    const float lnR = lerp1(T.el[mb + ei.i].x, T.el[mb + ei.i + 1].x, ei.f);
    const float s_maxe = lerp1(T.el2[mb2 + ei.i].x, T.el2[mb2 + ei.i + 1].x, ei.f) / rho0;
    const float maj = (a.pp.flags & 1) ? 0.f : __ldg(a.t.elmaj + ei.i);
    const bool ev = maj > 0.f;
    const uint32_t w1 = ev ? p.r.buf.y : p.r.buf.x;
    const float d_ev = ev ? -__logf(u01(p.r.buf.x)) / maj : 3.0e38f;
    p.r.n += ev ? 2u : 1u;
    float s = a.pp.d_maxs;
    int lim = 1;
    if (s_maxe < s) { s = s_maxe; lim = 2; }
    if (d_ev < s) { s = d_ev; lim = 3; }
    const float s1 = u01(w1) * s;
    const float Ef = E0 * (1.f - a.pp.f_maxe);
    const float Efull = csda_end2(T, m0, E0, __expf(lnR), range_to_lnE(T, m0, lnR), rho0 * s);
    float done, L = s1;
    int r;
    // up to the hinge, the deflection, the rest of the step: one copy of the voxel loop with one way out. With
    // a copy for each part, and a way out for each ending, a warp's lanes did not come together again after
    // the first part (8.7 lanes an instruction): 1e7 electrons of 15 MeV on the slab phantom took 182 ms at
    // 1.5 mm voxels and 136 at 2.5 mm, now 130 and 119; 5e6 at 1 mm 105, now 73.
#pragma unroll 1
    for (int part = 0;; ++part) {
        r = cross_segment(c, p, L, Ef, &done);
        if (part == 1 || r >= SEG_OUT) break;
        if (!(a.pp.flags & 2)) {
            EIdx em = e_index(0.5f * (E0 + Efull));
            float l1 = lerp1(T.el[mb + em.i].y, T.el[mb + em.i + 1].y, em.f);
            float cth = sample_ms(T, rho0 * (r == SEG_FLOOR ? done : s) * l1, p.r, k0, k1);
            float xphi = rng_u(p.r, k0, k1);
            rotate(p.u, p.v, p.w, cth, xphi);
        }
        if (r == SEG_FLOOR) break;
        L = s - s1;
    }
    if (r >= SEG_OUT) return segment_fate(r);
    if (r == SEG_FLOOR || lim != 3) return LIVE;
    // candidate hard event where the step ended
    if (vox_bad(c, p)) return GONE;
    const int v2 = p.ix + a.nx * (p.iy + a.ny * p.iz);
    const float rho = __ldg(a.density + v2);
    const int m = __ldg(a.material + v2);
    const EIdx e2 = e_index(p.E);
    const float4 A2 = T.el[m * MS4 + e2.i], B2 = T.el[m * MS4 + e2.i + 1];
    const float sM = p.E > 2.f * a.pp.w_cc ? rho * lerp1(A2.z, B2.z, e2.f) : 0.f;
    const float sB = p.E > a.pp.w_cb ? rho * lerp1(A2.w, B2.w, e2.f) : 0.f;
    const float tot = sM + sB;
    if (tot > maj * 1.00001f) count_rare(c, ST_VIOL, 1);
    if (rng_u(p.r, k0, k1) * maj < tot) {
        hard_event(c, p, m, sM, tot, sec);
        if (p.E < a.pp.e_abs_e) return ABSORBED;
    } else {
        count(c, ST_HARD_FICT);
    }
    return LIVE;
}

// The common tail: emits the pending secondary and carries out the lane's fate. A secondary below
// its absorption energy is deposited at the lane's voxel, as are an absorbed particle's energy and,
// below the photon cutoff, a positron's annihilation photons; a positron above it emits two photons
// of mc^2, back to back and isotropic, from its own stream.
template <class C>
__device__ __forceinline__ void finish(C& c, Lane& p, Pend& s, int fate)
{
    const TransportArgs& a = c.a;
    unsigned long long q = 0ull;
    const bool kerma = a.pp.flags & 8;
    int todo = 0;                                  // pushes: 1 the secondary, 2 the lane, 4 and 8 annihilation photons
    if (s.type >= 0) {
        if (s.type == PHOTON ? s.E >= a.pp.e_abs_g : s.E >= a.pp.e_abs_e && !kerma) todo = 1;
        else q = fx(s.E);
    }
    if (fate == ESCAPED) {
        count(c, ST_ESCAPED);
        add_energy(c, BE_ESC, fx(p.E));
    } else if (fate == MOVED) {
        todo |= 2;
    } else if (fate == ABSORBED) {
        q += p.E > 0.f ? fx(p.E) : 0ull;
        if (p.type == POSITRON) {
            count(c, ST_ANNIH);
            if (MC2F >= a.pp.e_abs_g) todo |= 12;
            else q += fx(2.f * MC2F);
        }
    }
    deposit_q(c, p, p.ix, p.iy, p.iz, q);
#pragma unroll 1
    while (todo) {
        if (!(todo & 1)) {
            if (todo & 2) {
                s.E = p.E; s.u = p.u; s.v = p.v; s.w = p.w;
                s.type = p.type;
                s.sub = p.r.sub;
                todo ^= 2;
            } else if (todo & 4) {
                float wc = 2.f * rng_u(p.r, a.key0, a.key1) - 1.f, xi = rng_u(p.r, a.key0, a.key1);
                float st = sqrtf(fmaxf(0.f, 1.f - wc * wc)), sp, cp;
                __sincosf(6.283185307179586f * xi, &sp, &cp);
                s.E = MC2F; s.u = st * cp; s.v = st * sp; s.w = wc;
                s.type = PHOTON;
                s.sub = child_sub(p.r.sub, p.r.n, 0);
                todo ^= 4;
            } else {
                s.u = -s.u; s.v = -s.v; s.w = -s.w;
                s.sub = child_sub(p.r.sub, p.r.n, 1);
                todo ^= 8;
            }
        } else {
            todo ^= 1;
        }
        push(c, s.type == PHOTON ? 0 : charged_stack(a, s.E), p, s.E, s.u, s.v, s.w, s.type, s.sub, 0u);
    }
}

// A warp moves the block's counts to the totals when its own iterations since the last time reach
// FLUSH_ITERS and when it ends: between two flushes a block's warps make at most 32 * 2^20 iterations
// of 32 lanes, so no 32-bit count of events (at most one of a kind per lane and step) wraps.
constexpr unsigned FLUSH_ITERS = 1u << 20;

__device__ __noinline__ void flush_stats(const TransportArgs& a, BlockStats& st, unsigned int* wc)
{
#pragma unroll 1
    for (int k = 0; k < ST_E_IN; ++k) {
        const unsigned v = atomicExch(&st.n[k], 0u);
        if (v) atomicAdd(a.stats + k, (unsigned long long)v);
    }
    // the halves one after the other: a carry that arrives between the two is added by the next flush
#pragma unroll 1
    for (int k = 0; k <= BE_MISS; ++k) {
        const unsigned lo = atomicExch(&st.e[k][0], 0u), hi = atomicExch(&st.e[k][1], 0u);
        const unsigned long long q = ((unsigned long long)hi << 32) + lo;
        if (q) atomicAdd(a.stats + ST_E_IN + k, q);
    }
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const unsigned v = atomicExch(wc + k, 0u);
        if (v) atomicAdd(a.stats + ST_WARP_ITERS + k, (unsigned long long)v);
    }
}

// A particle that never ends: dropped, with its energy counted.
template <class C>
__device__ __forceinline__ int step_limit(C& c, const Lane& p)
{
    atomicOr(c.a.err, ERR_LIMIT);
    count_rare(c, ST_DROPPED, 1);
    count_rare(c, ST_E_DROPPED, fx(p.E));
    return GONE;
}

// NREG: register cap per thread. More registers spill less; fewer registers let more
// warps share an SM (80: 3 x 256 threads, 64: 2 x 512, 56: 3 x 384 on GB300).
// PS: the source is a phase space (per-history records of mixed particle types); a separate
// instantiation, so that the analytic-source kernel carries none of its code.
// STEPS: the kind of electron steps, again an instantiation of the analytic-source kernel each.
// CROSS lets them cross voxel faces (the fixed-step variant). HELD takes apart what only a few lanes of a
// warp do after a step. A candidate hard event, whose code is as long as the step's, waits until HELD_MIN
// of the warp or a quarter of its lanes have one; those make no step meanwhile (6 % more iterations). A
// particle that ended without a secondary is put away when its lane is about to be refilled, which it
// waits for anyway. 5e6 electrons of 15 MeV on the half-slab phantom: 35.2 -> 32.3 ms (HELD_MIN 3: 33.9,
// 4: 33.1, 6 to 16: 32.5); 6e5 on water 3.71 -> 3.42 ms. The electrons of a photon beam have fewer
// events a step and lose by waiting (1e8 photons of 6 MV: 95.9 ms, 99.5 with it).
enum { PLAIN = 0, CROSS, HELD };
template <int BL, bool PS, int NREG, int STEPS = PLAIN>
__global__ void __maxnreg__(NREG) k_transport(const __grid_constant__ TransportArgs a)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ __align__(16) int s_top[MAX_WARPS][4];      // per warp: its stacks' tops (and a spare word)
    __shared__ BlockStats s_st;
    __shared__ unsigned long long s_time[MAX_WARPS][2];   // per warp: start, source seen exhausted
    __shared__ unsigned int s_wc[MAX_WARPS][4];           // per warp: iterations, photon / charged lane-steps
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int i = threadIdx.x; i < (int)(sizeof(BlockStats) / 4); i += blockDim.x) reinterpret_cast<unsigned*>(&s_st)[i] = 0u;
    const long long gw = (long long)blockIdx.x * (blockDim.x >> 5) + wib;
    // a resumed launch finishes what the warps of the launch before left on their photon stacks
    const int rest = a.left_in && *a.n_left_in ? a.left_in[gw] : 0;
    if (a.left_in && !__syncthreads_or(rest)) return;
    if (lane < 4) { s_top[wib][lane] = lane == 0 ? rest : 0; s_wc[wib][lane] = 0u; }
    SmemTables T = stage_tables(a.t, smem);   // ends with __syncthreads()
    if (lane == 0) { s_time[wib][0] = globaltimer_ns(); s_time[wib][1] = 0ull; }

    CtxT<BL> c{a, T, a.stacks + (size_t)gw * a.nstk * a.cap, s_top[wib], &s_st,
          1.f / a.dx, 1.f / a.dy, 1.f / a.dz, a.nx * a.dx, a.ny * a.dy, a.nz * a.dz};
    const unsigned lt = (1u << lane) - 1u;
    const int src_mode = a.src.particle == 0 ? 0 : 1;
    // a phase-space source mixes particle types: warps of either type draw from it, and a
    // primary of the other type goes to that type's stack like a secondary
    constexpr bool ps_src = PS && BL == ONE_BEAM;
    int mode = src_mode;
    bool src_done = a.count == 0 || wib >= a.src_warps;
    // with switch_high >= cap, switching on stack size is off (stacks may then overflow, which
    // is reported); otherwise a warp also switches when another stack nears its capacity
    const int emergency = a.switch_high < a.cap ? a.cap - 128 : 0x7FFFFFFF;
    // most iterations only step: nothing to schedule while few lanes are free and no stack is large
    const int plan_g = min(a.refill_g, 32 - a.switch_low), plan_e = min(a.refill_e, 32 - a.switch_low);
    const int plan_top = min(a.switch_high, emergency);
    // per-warp scheduler counters live in shared memory (iterations, photon and charged lane-steps):
    // none of them takes a register under the register cap
    unsigned int* wc = s_wc[wib];

    // modes (= stacks): 0 photons, 1 charged particles (at or above e_split when there are
    // three stacks), 2 charged particles below e_split
    bool active = false, just_switched = false;
    Lane p;
    int left = 0;                // photons this warp leaves to k_chains
    int fate = LIVE;
    Pend sec;
    sec.type = -1;
    float held = 0.f;            // > 0: the lane waits with a candidate hard event of this majorant
    for (;;) {
        __syncwarp();
        unsigned act = __ballot_sync(FULL, active);
        if constexpr (STEPS == HELD) {
            // what the last step emitted goes to its stack at once; particles that ended without emitting
            // anything keep until the free lanes are about to be refilled
            if (__any_sync(FULL, sec.type >= 0) ||
                (32 - __popc(act) >= (mode ? a.refill_e : a.refill_g) && __any_sync(FULL, fate != LIVE))) {
                if (fate != LIVE || sec.type >= 0) finish(c, p, sec, fate);
                fate = LIVE;
                sec.type = -1;
                __syncwarp();
            }
        } else {
            fate = LIVE;
            sec.type = -1;
        }
        const int4 tops = *reinterpret_cast<const int4*>(c.top);
        const int fullest = max(tops.x, max(tops.y, tops.z));
        bool settle = false;     // the waiting candidates now, no steps
        if (32 - __popc(act) >= (mode ? plan_e : plan_g) || fullest >= plan_top) {
            int top0 = min(tops.x, a.cap), top1 = min(tops.y, a.cap), top2 = a.nstk == 3 ? min(tops.z, a.cap) : 0;
            int nfree = 32 - __popc(act);
            // refill when enough lanes are free: the refill code runs on the free lanes only,
            // so waiting for several of them spreads its cost
            const int pool = mode == 1 ? top2 : (mode == 2 ? top1 : 0);   // the other charged stack
            if (nfree >= (mode ? a.refill_e : a.refill_g) || nfree == 32) {
                int topm = mode == 0 ? top0 : (mode == 1 ? top1 : top2);
                int rank = __popc(~act & lt);
                const int own = min(nfree, topm);
                // The classes are apart so that the lanes of a warp do alike steps (1e7 electrons of the slab
                // phantom: 69.8 ms, 76.3 with one class). Once the source is empty a lane without work costs
                // more than a mixed warp: 5e4 electrons of 15 MeV 1.08 ms with classes kept apart, 0.86 mixed.
                const int mix = src_done ? min(nfree - own, pool) : 0, take = own + mix;
                if (!active && rank < take) {
                    const bool o = rank < own;
                    pop_lane(c, o ? mode : 3 - mode, o ? topm - 1 - rank : pool - 1 - (rank - own), p);
                    active = true;
                }
                int want = min(nfree - take, a.src_share);
                if (want > 0 && (ps_src || mode == src_mode) && !src_done) {
                    unsigned long long base = 0;
                    if (lane == 0) base = atomicAdd(a.hist_counter, (unsigned long long)want);
                    base = __shfl_sync(FULL, base, 0);
                    if (base + want >= a.count) {
                        src_done = true;
                        if (lane == 0) s_time[wib][1] = globaltimer_ns();
                    }
                    int r2 = rank - take;
                    if (!active && r2 >= 0 && r2 < want && base + r2 < a.count) {
                        count(c, ST_HISTORIES);
                        bool in;
                        if constexpr (BL != ONE_BEAM) in = init_beamlet(a, base + r2, p);
                        else if constexpr (ps_src) in = init_phase_space(a, a.first + base + r2, p);
                        else in = init_primary(a, a.first + base + r2, p);
                        add_energy(c, in ? BE_IN : BE_MISS, fx(p.E));
                        if (!in) {
                            count(c, ST_MISSED);
                        } else {
                            const bool charged = p.type != PHOTON;
                            if (!(p.E >= (charged ? a.pp.e_abs_e : a.pp.e_abs_g)) || (charged && (a.pp.flags & 8))) fate = ABSORBED;
                            else if (ps_src && (charged ? charged_stack(a, p.E) : 0) != mode) fate = MOVED;
                            else active = true;
                        }
                    }
                }
                __syncwarp();
                if (lane == 0) {
                    c.top[mode] = topm - own;
                    if (mix) c.top[3 - mode] = pool - mix;
                    if (wc[0] >= FLUSH_ITERS) flush_stats(a, s_st, wc);
                }
                __syncwarp();
                if (mode == 0) top0 = topm - own;
                else if (mode == 1) top1 = topm - own, top2 -= mix;
                else top2 = topm - own, top1 -= mix;
                act = __ballot_sync(FULL, active);
                if (STEPS != HELD && __any_sync(FULL, fate != LIVE)) {
                    if (fate != LIVE) finish(c, p, sec, fate);
                    if (act == 0) continue;
                    fate = LIVE;
                    __syncwarp();
                }
            }
            int nact = __popc(act);
            const int topm = mode == 0 ? top0 : (mode == 1 ? top1 : top2);
            bool m_avail = topm > 0 || (src_done ? (mode == 1 ? top2 : (mode == 2 ? top1 : 0)) > 0 : ps_src || mode == src_mode);
            // the other mode: the fullest other stack that has work (or that the source feeds)
            int other = -1, topo = 0;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const int tk = k == 0 ? top0 : (k == 1 ? top1 : top2);
                if (k != mode && k < a.nstk && (tk > 0 || ((ps_src || k == src_mode) && !src_done)) &&
                    (other < 0 || tk > topo)) {
                    other = k;
                    topo = tk;
                }
            }
            const bool o_avail = other >= 0;
            if (nact == 0) {
                if (m_avail || (STEPS == HELD && __any_sync(FULL, fate != LIVE))) continue;
                if (o_avail) { mode = other; continue; }
                break;
            }
            bool sw = false;
            if (o_avail && !just_switched) {     // at most one switch between two steps
                // the other group must be strictly larger (or the source), so a switch is never undone at once
                if (!m_avail && nact <= a.switch_low && (topo > nact || (!ps_src && other == src_mode && !src_done)))
                    sw = true;
                else if (topo >= a.switch_high && topo >= 2 * (nact + topm)) sw = true;
                // the other stack is within one iteration's pushes (32 lanes x 3 secondaries, plus
                // 32 refilled primaries) of its capacity: switch before it can overflow
                else if (topo >= emergency && topo > topm) sw = true;
            }
            // few photons left in the warp, nothing to refill from and one of them in a long chain of
            // fictitious events: the warp ends and leaves them to k_chains, after the other stacks' work
            const bool chain = a.left_out && !sw && mode == 0 && !m_avail && nact <= CHAIN_LANES && !just_switched &&
                               __any_sync(FULL, active && p.steps >= CHAIN_STEPS && p.r.n < CHAIN_MAX_N) &&
                               !(STEPS == HELD && __any_sync(FULL, fate != LIVE));
            if (STEPS == HELD && sw && __any_sync(FULL, held > 0.f)) {
                settle = true;
            } else if (sw || chain) {
                if (active) {
                    push(c, mode ? charged_stack(a, p.E) : 0, p, p.E, p.u, p.v, p.w, p.type, p.r.sub, p.r.n);
                    active = false;
                }
                if (chain && !o_avail) { left = nact; break; }
                mode = other;
                just_switched = true;
                continue;
            }
            just_switched = false;
        }
        const unsigned step = STEPS != HELD ? act : settle ? 0u : act & ~__ballot_sync(FULL, held > 0.f);
        if (lane == 0) {
            atomicAdd(wc, 1u);
            atomicAdd(wc + (mode ? 2 : 1), (unsigned)__popc(step));
        }
        if constexpr (STEPS == HELD) {
            bool done = step >> lane & 1u;
            if (done) fate = mode ? charged_step<true>(c, p, sec, &held) : photon_step(c, p, sec);
            // (all of them while a stack is within one iteration's pushes of the point where the warp must
            // switch: it then switches at once)
            const int waits = __popc(__ballot_sync(FULL, held > 0.f));
            if (waits && (settle || waits >= HELD_MIN || 4 * waits >= __popc(act) || fullest >= emergency - 96)) {
                if (held > 0.f) {
                    fate = held_candidate(c, p, held, sec);
                    held = 0.f;
                    done = true;
                }
            }
            if (done && !(held > 0.f)) {
                if (fate == LIVE && ++p.steps > STEP_LIMIT) fate = step_limit(c, p);
                active = fate == LIVE;
                if (fate == GONE) fate = LIVE;       // nothing left to do
            }
        } else if (active) {
            if (mode) {
                if constexpr (STEPS == CROSS) fate = charged_step_cross(c, p, sec);
                else fate = charged_step<false>(c, p, sec, nullptr);
            } else {
                fate = photon_step(c, p, sec);
            }
            if (fate == LIVE && ++p.steps > STEP_LIMIT) fate = step_limit(c, p);
            active = fate == LIVE;
            if (fate > GONE || sec.type >= 0) finish(c, p, sec, fate);
        }
    }
    __syncwarp();
    if (lane == 0) {
        flush_stats(a, s_st, wc);
        if (a.left_out) {
            a.left_out[gw] = left;
            if (left) atomicAdd(a.n_left_out, 1ull);
        }
        // tail: how long this warp ran on its own stacks after the source ran dry
        const unsigned long long t_end = globaltimer_ns(), t0 = s_time[wib][0];
        const unsigned long long ts = s_time[wib][1] ? s_time[wib][1] : t0;
        atomicAdd(a.stats + ST_WARP_NS, t_end - t0);
        atomicAdd(a.stats + ST_TAIL_NS, t_end - ts);
        if (!a.left_in) {
            atomicAdd(a.stats + ST_WARPS, 1ull);
            atomicMax(a.stats + ST_T_START_INV, ~t0);
            if (s_time[wib][1]) atomicMax(a.stats + ST_T_SRC_INV, ~ts);
        }
        atomicMax(a.stats + ST_T_END, t_end);
    }
}

// Long Woodcock chains. A photon of a few tens of keV in air or lung flies against the majorant of
// the densest bone: hundreds to thousands of fictitious events in a row, one a step, in a warp whose
// other lanes have run dry; a short run then waited for a handful of such photons (half of the 3.6 ms
// of 1.3e6 6 MV photons on a CT-like 128^3 phantom). Between two real events the flights of a photon
// differ only in their random block and position, so a whole warp works on one photon here: lane j
// draws flight j of the next 32, all lanes follow the positions (the same chain of FMAs as the steps',
// so the same bits), each lane judges its own flight, and the photon moves past the fictitious ones
// before the first that is not; that one is left to photon_step in the resumed launch. One block per
// warp of the transport launch, one warp per photon; tables are read from global memory (L2).
__global__ void __launch_bounds__(32 * CHAIN_LANES) k_chains(const __grid_constant__ TransportArgs a)
{
    if (!*a.n_left_in) return;
    const int lane = threadIdx.x & 31, i = threadIdx.x >> 5;
    if (i >= a.left_in[blockIdx.x]) return;
    PRec* rec = a.stacks + (size_t)blockIdx.x * a.nstk * a.cap + i;
    PRec p = *rec;
    const float Lx = a.nx * a.dx, Ly = a.ny * a.dy, Lz = a.nz * a.dz;
    const float inv_dx = 1.f / a.dx, inv_dy = 1.f / a.dy, inv_dz = 1.f / a.dz;
    const EIdx ei = e_index(p.E);
    const float lnmaj = lerp1(__ldg(a.t.phmaj + ei.i), __ldg(a.t.phmaj + ei.i + 1), ei.f);
    if (lnmaj < -1e29f) return;
    const float mumax = __expf(lnmaj);
    unsigned flights = 0;
    for (int done = 32; done == 32 && p.n < CHAIN_MAX_N;) {
        const uint32_t blk = (p.n + 3u) >> 2;
        const uint4 b = philox4x32_10(make_uint4(blk + (uint32_t)lane, p.h0, p.h1, p.sub), a.key0, a.key1);
        const float s = -__logf(u01(b.x)) / mumax, u_real = u01(b.y);
        float x = p.x, y = p.y, z = p.z, mx = x, my = y, mz = z;
#pragma unroll 8
        for (int k = 0; k < 32; ++k) {
            const float sk = __shfl_sync(FULL, s, k);
            x = fmaf(sk, p.u, x);
            y = fmaf(sk, p.v, y);
            z = fmaf(sk, p.w, z);
            if (k == lane) { mx = x; my = y; mz = z; }
        }
        bool fict = mx >= 0.f && my >= 0.f && mz >= 0.f && mx <= Lx && my <= Ly && mz <= Lz;
        if (fict) {
            const int ix = min((int)(mx * inv_dx), a.nx - 1), iy = min((int)(my * inv_dy), a.ny - 1),
                      iz = min((int)(mz * inv_dz), a.nz - 1);
            const int vox = ix + a.nx * (iy + a.ny * iz);
            const float rho = __ldg(a.density + vox);
            const int m = __ldg(a.material + vox);
            const float mu = rho * __expf(lerp1(__ldg(&a.t.ph[m * NE + ei.i].x), __ldg(&a.t.ph[m * NE + ei.i + 1].x), ei.f));
            fict = u_real * mumax >= mu;
        }
        const unsigned stop = __ballot_sync(FULL, !fict);
        done = stop ? __ffs(stop) - 1 : 32;
        if (done) {
            p.x = __shfl_sync(FULL, mx, done - 1);
            p.y = __shfl_sync(FULL, my, done - 1);
            p.z = __shfl_sync(FULL, mz, done - 1);
            p.n = (blk + (uint32_t)done) << 2;
            flights += (unsigned)done;
        }
    }
    __syncwarp();                              // every lane has read the record
    if (lane == 0) {
        rec->x = p.x; rec->y = p.y; rec->z = p.z;
        rec->n = p.n;
        atomicAdd(a.stats + ST_FICT, (unsigned long long)flights);
        atomicAdd(a.stats + ST_LANES_PHOTON, (unsigned long long)flights);
    }
}

}  // namespace

size_t transport_smem_bytes(int n_mat) { return smem_table_bytes(n_mat); }

namespace {
constexpr unsigned long long SRC_LANES = 28;
// Histories a warp from which an electron beam's run holds its hard events: below, a run is the chain of
// steps of its last particles, which waiting lengthens. 15 MeV with 4864 warps, without and with it, in ms:
//   histories                          5e4   1e5   2e5   3e5   4e5   6e5   1e6    2e6
//   water 61 x 61 x 60 at 0.5 cm       0.72  0.92  1.54  2.02  2.58  3.69  5.80  11.05
//                                      0.74  0.95  1.50  1.96  2.42  3.38  5.24   9.85
//   half-slab 120^3 at 0.25 cm         1.37  1.68  2.52  3.20  3.95  5.29  8.05  14.79
//                                      1.41  1.74  2.56  3.14  3.77  5.05  7.50  13.64
constexpr unsigned long long HELD_HISTORIES = 64;

template <int BL, bool PS, int R, int STEPS = PLAIN>
cudaError_t launch_variant(const TransportArgs& a, int blocks, int threads, size_t smem, cudaStream_t s)
{
    cudaError_t e =
        cudaFuncSetAttribute(k_transport<BL, PS, R, STEPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    k_transport<BL, PS, R, STEPS><<<blocks, threads, smem, s>>>(a);
    return cudaGetLastError();
}

template <int BL, bool PS, int R>
int occupancy(int threads, size_t smem)
{
    cudaFuncSetAttribute(k_transport<BL, PS, R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_transport<BL, PS, R>, threads, smem) != cudaSuccess)
        return 0;
    return n;
}

template <int STEPS, int BL = ONE_BEAM, bool PS = false>
cudaError_t launch_steps(const TransportArgs& a, int blocks, int threads, size_t smem, cudaStream_t s, int nreg)
{
    if (nreg == 56) return launch_variant<BL, PS, 56, STEPS>(a, blocks, threads, smem, s);
    if (nreg == 64) return launch_variant<BL, PS, 64, STEPS>(a, blocks, threads, smem, s);
    return launch_variant<BL, PS, 80, STEPS>(a, blocks, threads, smem, s);
}
}  // namespace

bool transport_nreg_supported(int nreg) { return nreg == 56 || nreg == 64 || nreg == 80; }

int transport_max_blocks_per_sm(int threads, size_t smem, int nreg)
{
    occupancy<BEAMLETS_DENSE, false, 56>(threads, smem);
    occupancy<BEAMLETS_HASH, false, 56>(threads, smem);   // sets the shared-memory attribute of every variant
    occupancy<BEAMLETS_DENSE, false, 64>(threads, smem);
    occupancy<BEAMLETS_HASH, false, 64>(threads, smem);
    occupancy<BEAMLETS_DENSE, false, 80>(threads, smem);
    occupancy<BEAMLETS_HASH, false, 80>(threads, smem);
    occupancy<ONE_BEAM, true, 56>(threads, smem);
    occupancy<ONE_BEAM, true, 64>(threads, smem);
    occupancy<ONE_BEAM, true, 80>(threads, smem);
    cudaFuncSetAttribute(k_transport<ONE_BEAM, false, 56, CROSS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_transport<ONE_BEAM, false, 56, HELD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_transport<ONE_BEAM, false, 64, CROSS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_transport<ONE_BEAM, false, 64, HELD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_transport<ONE_BEAM, false, 80, CROSS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    cudaFuncSetAttribute(k_transport<ONE_BEAM, false, 80, HELD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (nreg == 56) return occupancy<ONE_BEAM, false, 56>(threads, smem);
    if (nreg == 64) return occupancy<ONE_BEAM, false, 64>(threads, smem);
    return occupancy<ONE_BEAM, false, 80>(threads, smem);
}

static cudaError_t launch_one(const TransportArgs& a, int blocks, int threads, size_t smem, cudaStream_t s, int nreg)
{
    if (a.pp.flags & FLAG_CROSS_VOXELS) {
        // voxel-crossing electron steps: analytic single-beam source only (callers check)
        if (a.beamlets || a.ps) return cudaErrorInvalidValue;
        return launch_steps<CROSS>(a, blocks, threads, smem, s, nreg);
    }
    if (a.beamlets)
        return a.bl_dense ? launch_steps<PLAIN, BEAMLETS_DENSE, false>(a, blocks, threads, smem, s, nreg)
                          : launch_steps<PLAIN, BEAMLETS_HASH, false>(a, blocks, threads, smem, s, nreg);
    if (a.ps) return launch_steps<PLAIN, ONE_BEAM, true>(a, blocks, threads, smem, s, nreg);
    if (a.held) return launch_steps<HELD>(a, blocks, threads, smem, s, nreg);
    return launch_steps<PLAIN, ONE_BEAM, false>(a, blocks, threads, smem, s, nreg);
}

cudaError_t launch_transport(const TransportArgs& args, int blocks, int threads, size_t smem, cudaStream_t s, int nreg)
{
    TransportArgs a = args;
    // A run with fewer histories than lanes is spread over all blocks, and in each over as few warps as
    // hold its share at SRC_LANES a warp: whole blocks stay without work when every warp draws 32 at once,
    // and a step of 10 lanes costs a warp as much as one of 30 (5e4 electrons of 15 MeV on 152 blocks of 32
    // warps: 12 warps with 28 lanes 0.71 ms, 24 with 14 0.81, 32 with 11 0.84; 1e5 photons 0.82, 0.83, 0.85).
    // Warps in fours, as a block's warps are dealt out to the four schedulers in turn.
    const unsigned long long warps = (unsigned long long)blocks * (threads / 32), per = (a.count + blocks - 1) / blocks;
    const unsigned long long busy = (per + SRC_LANES - 1) / SRC_LANES;
    a.src_warps = (int)std::min<unsigned long long>(threads / 32, (busy + 3) / 4 * 4);
    a.src_share = (int)std::min<unsigned long long>(32, (per + a.src_warps - 1) / a.src_warps);
    a.held = a.src.particle == 1 && !a.beamlets && !a.ps && a.count >= HELD_HISTORIES * warps;
    int* left = a.left_out;                      // one count per warp; null: no room for it, every warp finishes its photons
    a.n_left_out = a.hist_counter + 1;
    cudaError_t e = launch_one(a, blocks, threads, smem, s, nreg);
    if (!left || e != cudaSuccess) return e;
    // the photons that warps left in long chains (usually none: both launches then return at once)
    a.left_in = left;
    a.n_left_in = a.hist_counter + 1;
    a.left_out = nullptr;
    a.count = 0;
    k_chains<<<(unsigned)warps, 32 * CHAIN_LANES, 0, s>>>(a);
    e = cudaGetLastError();
    return e != cudaSuccess ? e : launch_one(a, blocks, threads, smem, s, nreg);
}

}  // namespace ocmc
