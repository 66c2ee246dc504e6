// reed_ion.cuh -- the track stepper of the ion-target-only model (target
// model NONE): one warp follows one track.  (Wide runs that would leave an SM's
// warps idle get a block of threads per track, see ion_by_block.)
//
// Without target-target forces an atom that the ion has not come near is at
// rest and stays at rest, so a step concerns three sets only:
//   * the atoms that move (the ion has pushed them) or lie within the cutoff
//     plus a skin of the ion: the track's list, some 60 of a window's 216 or
//     90 of 324 atoms.  It is rebuilt from the whole window when the ion has
//     gone the skin's length since the last build, and after a window move.
//     Atoms at rest do not move, so nothing else can invalidate it;
//   * those of the list within the cutoff now (about 26 or 38), collected
//     while the list is kicked and drifted, so that the pair function runs
//     once on nearly full warps;
//   * the ion itself, whose state is held in registers by every lane (FP64
//     position and time: one lane each, so that a step adds them all with two
//     FP64 instructions).
//
// Results do not depend on which lane evaluates which atom: an atom's pair
// term (g, d) is kept in shared memory at the atom's index, and the sums over
// atoms are taken by `vt` virtual threads -- thread t adds atoms t, t + vt,
// t + 2 vt ... in that order, 32 consecutive threads are added by a butterfly,
// the groups of 32 in order -- the summation order of a block of vt threads
// with one atom per thread and pass.  threads_per_track selects vt.
//
// What bounds a step: instruction issue and its latency -- some 850 warp
// instructions, 4200 cycles in the mixed form when a track runs alone and 5200
// with 16 on an SM, whose issue slots are then 62 % busy -- and in the FP64 form
// the FP64 pipe (64 % busy with four tracks on an SM).  A block of 64 threads that
// tested every atom of the window in each step, with one thread's ion update
// between two barriers, took 1700 instructions.  Measured on whole runs (block
// of 64 -> one warp): 32 B ions of 1 keV 17.3 -> 11.8 ms, 3001 of 10 keV 200 -> 114
// ms, 500 of 1 keV in FP64 300 -> 98 ms, 131 Kr of 85 MeV (10^4 steps each) 51.1
// -> 27.2 ms.
#pragma once

#include <type_traits>

#include "reed_track.cuh"

// The list's skin, A: the list is rebuilt every ten steps of 0.05 A.
#define REED_ION_SKIN 0.5

// Shared memory of a track that keeps no adjoint (TrackShared has the same
// members for the adjoint's CTAs).
template <typename R> struct IonShared {
    IonState<R> ion;           // id, keys; complete only in records
    double thr[REED_MAX_THR];  // this track's cloning depths (frozen while it runs)
    int nthr, src, top, slot;
    int was_busy;              // this CTA is counted among its SM's tracks
    int need_count, active_count, nhit0;   // build_ion_list: entries of the list, integrated atoms, hits
    long long pidx;
    unsigned long long cnt[ION_NCOUNT];
};

template <typename R, bool ADJ> struct IonLayout {
    using Base = Layout<R, REED_TT_NONE>;
    static __host__ __device__ size_t head_bytes()
    {
        return Base::align(ADJ ? sizeof(TrackShared<R>) : sizeof(IonShared<R>));
    }
    // pos, vel, pair terms; the adjoint's xbar, vbar; the list and the hits
    static __host__ __device__ size_t total(int na)
    {
        return head_bytes() + (ADJ ? 5 : 3) * Base::align(sizeof(V4<R>) * na) + 2 * Base::align(sizeof(uint16_t) * na);
    }
};

// The ion during the step loop, in registers: the same values in every lane,
// except acc.
template <typename R> struct IonRegs {
    R v[3], vlo[3], f[3];
    R rel[3];              // position relative to the anchor corner
    R rho, vmax2, pmax, dt;
    R zthr, zback, zsurf;  // next cloning depth, backscatter plane, surface in the anchor frame
    double acc;            // lanes 0-2: position, lane 3: time
    int A[3];
    int level;
    long long steps;
};

template <typename R> __device__ __forceinline__ R lane_of(const R x[3], int lane)
{
    return lane == 0 ? x[0] : (lane == 1 ? x[1] : x[2]);
}
__device__ __forceinline__ int lane_of(const int x[3], int lane) { return lane == 0 ? x[0] : (lane == 1 ? x[1] : x[2]); }

template <typename R> __device__ __forceinline__ void pack_ion(const IonRegs<R>& I, IonState<R>& s, int lane)
{
    if (lane < 3) s.x[lane] = I.acc;
    if (lane == 3) s.t = I.acc;
    if (lane == 0) {
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            s.v[d] = I.v[d];
            s.vlo[d] = I.vlo[d];
            s.f[d] = I.f[d];
            s.A[d] = I.A[d];
        }
        s.rho = I.rho;
        s.vmax2 = I.vmax2;
        s.pmax = I.pmax;
        s.steps = I.steps;
        s.level = I.level;
    }
    __syncwarp();
}

template <typename R> __device__ __forceinline__ void unpack_ion(IonRegs<R>& I, const IonState<R>& s, int lane)
{
    I.acc = lane < 3 ? s.x[lane] : s.t;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        I.v[d] = s.v[d];
        I.vlo[d] = s.vlo[d];
        I.f[d] = s.f[d];
        I.A[d] = s.A[d];
    }
    I.rho = s.rho;
    I.vmax2 = s.vmax2;
    I.pmax = s.pmax;
    I.steps = s.steps;
    I.level = s.level;
}

// Depth of the ion for the cloning depths (see track_depth), in every lane.
template <typename R> __device__ __forceinline__ double regs_depth(const DevParams& P, const IonRegs<R>& I)
{
    const double z = __shfl_sync(0xffffffffu, I.acc, 2);
    if (!P.bulk) return z;
    const double x = __shfl_sync(0xffffffffu, I.acc, 0), y = __shfl_sync(0xffffffffu, I.acc, 1);
    return sqrt(__dadd_rn(__dadd_rn(__dmul_rn(x, x), __dmul_rn(y, y)), __dmul_rn(z, z)));
}

// Anchor-frame quantities (see set_frame).  On a bulk target zthr is the
// square of the next cloning distance, reduced by more than the rounding of
// an FP32 position: the FP64 distance is taken only from there on.
template <typename R>
__device__ __forceinline__ void regs_frame(const DevParams& P, IonRegs<R>& I, const double* thr, int nthr, int lane)
{
    const double mine = I.acc;
    // (x and y in one rounding, z in two: the product is the anchor's depth z0)
    const double an = (double)lane_of(I.A, lane), z0 = __dmul_rn((double)I.A[2], P.a);
    const R r = R(lane == 2 ? __dsub_rn(mine, z0) : fma(-an, P.a, mine));
#pragma unroll
    for (int d = 0; d < 3; ++d) I.rel[d] = __shfl_sync(0xffffffffu, r, d);
    if (P.bulk) {
        I.zback = R(-1e30);
        I.zsurf = R(-1e30);
        const double t = I.level < nthr ? max(thr[I.level] * (1.0 - 1e-5) - 0.1, 0.0) : 1e15;
        I.zthr = R(t * t);
        return;
    }
    I.zthr = I.level < nthr ? R(thr[I.level] - z0) : R(1e30);
    I.zback = R(-P.rc - z0);
    I.zsurf = R(-z0);
}

template <typename R> __device__ __forceinline__ R regs_drag(const HotParams<R>& H, const IonRegs<R>& I)
{
    if (I.rel[2] < I.zsurf) return R(0);
    return H.gamma * (R(1) + H.s_loc * (I.rho * H.rho0_inv - R(1)));
}

// One half kick of the ion at the velocity it has (see ion_step).
template <typename R> __device__ __forceinline__ void regs_kick(const HotParams<R>& H, IonRegs<R>& I)
{
    const R kd = regs_drag<R>(H, I);
    const R h = R(0.5) * I.dt * H.invM1;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        // (in these roundings on every path: a track's bits depend on them)
        add_velocity<R>(I.v[d], I.vlo[d], h * add_rn(I.f[d], mul_rn(-kd, I.v[d])));
    }
}

// Start of a step: dt, the ion's half kick and drift, window anchor check
// (see ion_step).  Returns whether the window moves; Aold is the anchor before.
template <typename R>
__device__ __forceinline__ bool regs_prologue(const DevParams& P, const HotParams<R>& H, IonRegs<R>& I, int Aold[3],
                                              const double* thr, int nthr, int lane)
{
    const R v2 = dist2(I.v[0], I.v[1], I.v[2]);
    const R vmax = sqrt(max(v2, I.vmax2));
    R dt = H.dt_max;
    if (vmax * dt > H.dx_max) dt = H.dx_max / vmax;
    if (H.de_max > R(0)) {
        const R pw = max(fabs(dot3(I.f[0], I.f[1], I.f[2], I.v[0], I.v[1], I.v[2])), I.pmax);
        if (pw * dt > H.de_max) {
            dt = H.de_max / pw;
            if (vmax * dt < H.dx_min) dt = H.dx_min / vmax;
        }
    }
    I.dt = dt;
    regs_kick<R>(H, I);
    R dx[3];
    bool out[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        dx[d] = dt * I.v[d];
        I.rel[d] += dx[d];
        Aold[d] = I.A[d];
        out[d] = I.rel[d] >= H.anchor_hi || I.rel[d] < H.anchor_lo;
    }
    if (sizeof(R) == 8) I.acc = fma((double)dt, lane < 3 ? (double)lane_of(I.v, lane) : 0.0, I.acc);
    else I.acc += lane < 3 ? (double)lane_of(dx, lane) : 0.0;
    if (!(out[0] || out[1] || out[2])) return false;
    const int An = (int)floor(I.acc / P.a + P.anchor_shift);
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        const int a = __shfl_sync(0xffffffffu, An, d);
        if (out[d]) I.A[d] = a;
    }
    regs_frame<R>(P, I, thr, nthr, lane);
    return true;
}

// The force on an atom from its pair term.
template <typename R> __device__ __forceinline__ void pair_term_force(const V4<R>& t, R& fx, R& fy, R& fz)
{
    fx = -(t.x * t.y);
    fy = -(t.x * t.z);
    fz = -(t.x * t.w);
}

// A track's window in shared memory.
template <typename R> struct IonWin {
    V4<R>* pos;      // relative to the anchor corner; w: species and flags
    V4<R>* vel;      // w: the atom's local-density weight at the ion (0 outside the cutoff)
    V4<R>* term;     // pair term with the ion: g = dU/dr / r and d = x_atom - x_ion; 0 outside the cutoff
    uint16_t* list;  // atoms that move or lie within the cutoff plus the skin
    uint16_t* hit;   // those within the cutoff
    int nlist, nhit;
    R bx, by, bz;    // the ion's position when the list was built
    __device__ IonWin(unsigned char* base, size_t head, int na, bool adj)
    {
        const size_t ab = Layout<R, REED_TT_NONE>::align(sizeof(V4<R>) * na);
        pos = reinterpret_cast<V4<R>*>(base + head);
        vel = reinterpret_cast<V4<R>*>(base + head + ab);
        term = reinterpret_cast<V4<R>*>(base + head + 2 * ab);
        list = reinterpret_cast<uint16_t*>(base + head + (adj ? 5 : 3) * ab);
        hit = list + Layout<R, REED_TT_NONE>::align(sizeof(uint16_t) * na) / sizeof(uint16_t);
        nlist = nhit = 0;
        bx = by = bz = R(0);
    }
};

// The list and the hits from the whole window (one warp), after the window
// move from Aold to A when `shift`.  `clear`: atoms outside the cutoff have no
// pair term any more (not at the start of a clone, whose first half kick takes
// the terms of the record).  Returns the largest speed^2 of the integrated
// atoms outside the cutoff in this lane; the counts go to S.  Out of line and
// with arguments by value: it runs every ten steps or more and would else keep
// the stepping code's registers in memory.
template <typename R, typename Head>
__device__ __noinline__ R build_ion_list(const DevParams& P, const DevBuf& B, Head* S, V4<R>* pos, V4<R>* vel,
                                         V4<R>* term, uint16_t* list, uint16_t* hit, R x, R y, R z, int ax, int ay,
                                         int az, int ox, int oy, int oz, int level, bool shift, bool clear)
{
    const HotParams<R>& H = hot<R>(P);
    const int lane = threadIdx.x & 31;
    const uint64_t key = S->ion.key;
    const int A[3] = {ax, ay, az}, Aold[3] = {ox, oy, oz};
    const R rl = sqrt(H.rc2) + R(REED_ION_SKIN), rl2 = rl * rl;
    const V4<R> none = {R(0), R(0), R(0), R(0)};
    R vm = R(0);
    int nl = 0, nh = 0, nact = 0;
    for (int i0 = 0; i0 < P.na; i0 += 32) {
        const int i = i0 + lane;
        bool in_list = false, in_range = false, act = false;
        if (i < P.na) {
            V4<R> p = pos[i], v = vel[i], t = term[i];
            if (shift) {
                const V4<R> p0 = p, v0 = v;
                if (reanchor_atom<R>(P, H, key, i, Aold, A, p, v, t))
                    deposit_damage<R>(P, B, p0, v0, Aold, ldexp(1.0, -level));
                pos[i] = p;
                vel[i] = v;
                term[i] = t;
            }
            if (is_present(p)) {
                act = is_active(p);
                const R dx = p.x - x, dy = p.y - y, dz = p.z - z;
                const R r2 = dist2(dx, dy, dz);
                const bool moving = act && (v.x != R(0) || v.y != R(0) || v.z != R(0));
                in_range = r2 < H.rc2;
                // (an atom whose force underflows can still have a density weight)
                const bool term_on = t.x != R(0) || v.w != R(0);
                in_list = in_range || r2 < rl2 || moving || term_on;
                if (!in_range) {
                    if (clear && term_on) {
                        term[i] = none;
                        vel[i].w = R(0);
                    }
                    if (moving) vm = max(vm, dist2(v.x, v.y, v.z));
                }
            }
        }
        const unsigned bl = __ballot_sync(0xffffffffu, in_list), bh = __ballot_sync(0xffffffffu, in_range);
        const unsigned below = (1u << lane) - 1u;
        if (in_list) list[nl + __popc(bl & below)] = (uint16_t)i;
        if (in_range) hit[nh + __popc(bh & below)] = (uint16_t)i;
        nl += __popc(bl);
        nh += __popc(bh);
        nact += __popc(__ballot_sync(0xffffffffu, act));
    }
    if (lane == 0) {
        S->need_count = nl;
        S->active_count = nact;
        S->nhit0 = nh;
    }
    __syncwarp();
    return vm;
}

// Half kick, drift and (unless the list is about to be rebuilt) the cutoff
// test of one listed atom; returns whether it lies within the cutoff.
template <typename R>
__device__ __forceinline__ bool ion_move_atom(const HotParams<R>& H, IonWin<R>& W, const IonRegs<R>& I, int i, V4<R> p,
                                              V4<R> v, const V4<R>& t, R hdt, bool test, R& vm)
{
    const bool act = is_active(p);
    if (act) {
        R fx, fy, fz;
        pair_term_force(t, fx, fy, fz);
        const R k = hdt * of_species(H.invM2, p);
        v.x = fma(k, fx, v.x);
        v.y = fma(k, fy, v.y);
        v.z = fma(k, fz, v.z);
        p.x = fma(I.dt, v.x, p.x);
        p.y = fma(I.dt, v.y, p.y);
        p.z = fma(I.dt, v.z, p.z);
        W.pos[i] = p;
    }
    if (!test) {
        if (act) W.vel[i] = v;
        return false;
    }
    const R dx = p.x - I.rel[0], dy = p.y - I.rel[1], dz = p.z - I.rel[2];
    const R r2 = dist2(dx, dy, dz);
    const bool in = r2 < H.rc2;
    if (!in) {
        if (t.x != R(0)) W.term[i] = {R(0), R(0), R(0), R(0)};   // it has just left the cutoff
        v.w = R(0);
        if (act) vm = max(vm, dist2(v.x, v.y, v.z));
    }
    W.vel[i] = v;
    return in;
}

// Pair terms of the atoms within the cutoff and, with KICK, their second half
// kick; vm and pm as in the force pass of the other models.
template <typename R, bool KICK>
__device__ __forceinline__ void ion_pair_pass(const DevParams& P, const HotParams<R>& H, IonWin<R>& W,
                                              const IonRegs<R>& I, R hdt, R& vm, R& pm)
{
    for (int e = threadIdx.x & 31; e < W.nhit; e += 32) {
        const int i = W.hit[e];
        const V4<R> p = W.pos[i];
        const R dx = p.x - I.rel[0], dy = p.y - I.rel[1], dz = p.z - I.rel[2];
        const R r2 = dist2(dx, dy, dz);
        R U, rw;
        const R g = ion_pair<R>(H, P.spline_on, P.rho_on, is_second(p), r2, U, rw);
        const V4<R> t = {g, dx, dy, dz};
        W.term[i] = t;
        V4<R> v = W.vel[i];
        v.w = rw;
        if (KICK && is_active(p)) {
            R fx, fy, fz;
            pair_term_force(t, fx, fy, fz);
            const R kk = hdt * of_species(H.invM2, p);
            v.x = fma(kk, fx, v.x);
            v.y = fma(kk, fy, v.y);
            v.z = fma(kk, fz, v.z);
            vm = max(vm, dist2(v.x, v.y, v.z));
            if (H.de_max > R(0)) pm = max(pm, fabs(dot3(fx, fy, fz, v.x, v.y, v.z)));
        }
        W.vel[i] = v;
    }
    __syncwarp();
}

// Force on the ion and the local density: the sums of the pair terms by vt
// virtual threads (see the head of this file).  Two groups of 32 threads at a
// time: the first butterfly stage leaves each group to one half of the warp,
// the next two leave one sum to each four lanes, so that a sum of 64 terms
// costs 9 shuffles and not 40.
template <typename R>
__device__ __forceinline__ void ion_sums(const DevParams& P, const IonWin<R>& W, IonRegs<R>& I, int vt)
{
    constexpr unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
    R acc = R(0);   // lanes 0-3: fx, 4-7: fy, 8-11: fz, 12-15: density (and the same in the upper half)
    const bool two = vt > 32;
    const V4<R> none = {R(0), R(0), R(0), R(0)};
    for (int t0 = 0; t0 < vt; t0 += 64) {
        R s0[4] = {R(0), R(0), R(0), R(0)}, s1[4] = {R(0), R(0), R(0), R(0)};
        // (an absent atom adds 0 * 0, which changes no sum)
#pragma unroll 3
        for (int i = t0 + lane; i - lane < P.na; i += vt) {
            const bool on0 = i < P.na, on1 = two && i + 32 < P.na;
            const V4<R> a = on0 ? W.term[i] : none, b = on1 ? W.term[i + 32] : none;
            s0[0] = fma(a.x, a.y, s0[0]);
            s0[1] = fma(a.x, a.z, s0[1]);
            s0[2] = fma(a.x, a.w, s0[2]);
            s1[0] = fma(b.x, b.y, s1[0]);
            s1[1] = fma(b.x, b.z, s1[1]);
            s1[2] = fma(b.x, b.w, s1[2]);
            if (P.rho_on) {
                s0[3] += on0 ? W.vel[i].w : R(0);
                s1[3] += on1 ? W.vel[i + 32].w : R(0);
            }
        }
        R k4[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const R other = __shfl_xor_sync(FULL, b4 ? s0[c] : s1[c], 16);
            k4[c] = (b4 ? s1[c] : s0[c]) + other;
        }
        R k2[2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
            const R other = __shfl_xor_sync(FULL, b3 ? k4[c] : k4[c + 2], 8);
            k2[c] = (b3 ? k4[c + 2] : k4[c]) + other;
        }
        R k = (b2 ? k2[1] : k2[0]) + __shfl_xor_sync(FULL, b2 ? k2[0] : k2[1], 4);
        k += __shfl_xor_sync(FULL, k, 2);
        k += __shfl_xor_sync(FULL, k, 1);
        const R other = __shfl_xor_sync(FULL, k, 16);
        acc += b4 ? other : k;
        if (two) acc += b4 ? k : other;
    }
    I.f[0] = __shfl_sync(FULL, acc, 0);
    I.f[1] = __shfl_sync(FULL, acc, 4);
    I.f[2] = __shfl_sync(FULL, acc, 8);
    I.rho = __shfl_sync(FULL, acc, 12);
}

// The window in the clone-record format.  As checkpoint of an adjoint run
// (FORCES) the third array holds the atoms' forces, which its reverse pass
// starts from, else the pair terms.
template <typename R, bool FORCES>
__device__ __forceinline__ void save_window(const DevParams& P, const V4<R>* pos, const V4<R>* vel, const V4<R>* term,
                                            unsigned char* rec)
{
    V4<R>* g = reinterpret_cast<V4<R>*>(rec + Layout<R, REED_TT_NONE>::align(sizeof(IonState<R>)));
    for (int i = threadIdx.x & 31; i < P.na; i += 32) {
        V4<R> v = vel[i], t = term[i];
        if (FORCES) {
            V4<R> f = {R(0), R(0), R(0), R(0)};
            if (t.x != R(0)) pair_term_force(t, f.x, f.y, f.z);
            t = f;
            v.w = R(0);
        }
        g[i] = pos[i];
        g[P.na + i] = v;
        g[2 * P.na + i] = t;
    }
}

template <typename R>
__device__ __forceinline__ void load_window(const DevParams& P, IonWin<R>& W, const unsigned char* rec)
{
    // (records may have been written by another SM: read them from L2)
    const uint4* g = reinterpret_cast<const uint4*>(rec + Layout<R, REED_TT_NONE>::align(sizeof(IonState<R>)));
    const int m = P.na * (int)(sizeof(V4<R>) / sizeof(uint4));
    uint4 *pos = reinterpret_cast<uint4*>(W.pos), *vel = reinterpret_cast<uint4*>(W.vel),
          *term = reinterpret_cast<uint4*>(W.term);
    for (int i = threadIdx.x & 31; i < m; i += 32) {
        pos[i] = __ldcg(g + i);
        vel[i] = __ldcg(g + m + i);
        term[i] = __ldcg(g + 2 * m + i);
    }
}

template <typename R> __device__ __forceinline__ void load_header(IonState<R>& s, const unsigned char* rec)
{
    const uint4* h = reinterpret_cast<const uint4*>(rec);
    uint4* d = reinterpret_cast<uint4*>(&s);
    for (int k = threadIdx.x & 31; k < (int)(sizeof(IonState<R>) / sizeof(uint4)); k += 32) d[k] = __ldcg(h + k);
}

// The next track of this warp into S and W: the top of its clone stack, a
// primary, or a clone from the pool (see reed_track_kernel).  Returns its
// source, SRC_NONE when there is no more work.
template <typename R, typename Head>
__device__ int acquire_track(const DevParams& P, const DevBuf& B, Head* S, IonWin<R>& W, const unsigned char* stack,
                             int lane)
{
    if (lane == 0) {
        S->nthr = P.nthr;
        for (int k = 0; k < P.nthr; ++k) S->thr[k] = P.thr_from_device ? B.thr[k] : P.thr[k];
        if (S->top > 0) {
            S->src = SRC_CLONE;
        } else if (P.stop_after > 0 && (long long)(*(volatile unsigned long long*)B.finished) >= P.stop_after) {
            S->src = SRC_NONE;   // enough tracks collected: hand out no more primaries
        } else if (B.pool && (long long)blockIdx.x >= P.n_primaries) {
            S->src = SRC_NONE;   // the first CTAs, which are spread over the SMs, take one primary each
        } else {
            const unsigned long long k = atomicAdd(B.next, 1ull);
            S->pidx = (long long)k;
            S->src = ((long long)k < P.n_primaries) ? SRC_PRIMARY : SRC_NONE;
        }
        // Tracks followed on each SM.  A clone is best taken where few others
        // share the SM, so an idle CTA lets a record lie for one poll per track
        // on its SM; a CTA of an idle SM takes it at once.
        unsigned smid;
        asm("mov.u32 %0, %%smid;" : "=r"(smid));
        unsigned* busy = B.pool ? &B.pool_ctl[3 + smid % REED_POOL_SMS] : nullptr;
        if (B.pool && S->was_busy != (S->src != SRC_NONE)) {
            if (S->src != SRC_NONE) atomicAdd(busy, 1u);
            else atomicSub(busy, 1u);
            S->was_busy = S->src != SRC_NONE;
        }
        if (S->src == SRC_NONE && B.pool && P.nthr > 0) {   // (no clones without cloning depths)
            unsigned seen = 0;
            // out of work: take a donated clone, or stop once every CTA is
            // idle and no record is reserved or held
            bool idle = false;
            for (long long it = 0;; ++it) {
                seen = *(volatile unsigned*)&B.pool_ctl[2] > 0u ? seen + 1u : 0u;
                const int sl =
                    seen && seen > *(volatile unsigned*)busy ? pool_claim(B, POOL_FULL, POOL_READING) : -1;
                if (sl >= 0) {
                    atomicAdd(busy, 1u);
                    S->was_busy = 1;
                    atomicSub(&B.pool_ctl[2], 1u);
                    if (idle) atomicSub(&B.pool_ctl[0], 1u);
                    S->slot = sl;
                    S->src = SRC_STOLEN;
                    break;
                }
                if (!idle) {
                    atomicAdd(&B.pool_ctl[0], 1u);
                    idle = true;
                }
                if (*(volatile unsigned*)&B.pool_ctl[0] >= gridDim.x && *(volatile unsigned*)&B.pool_ctl[1] == 0u) break;
                if (it >= P.pool_polls) {
                    atomicOr(B.status, ERR_TIMEOUT);
                    break;
                }
                __nanosleep(it < 64 ? 500u : 4000u);
            }
        }
    }
    __syncwarp();
    const int src = S->src;
    if (src == SRC_NONE) return src;
    if (src == SRC_PRIMARY) {
        if (lane == 0) launch_primary<R>(P, S->ion, S->pidx);
        __syncwarp();
        const uint64_t key = S->ion.key;
        const int A[3] = {S->ion.A[0], S->ion.A[1], S->ion.A[2]};
        for (int i = lane; i < P.na; i += 32) {
            V4<R> p, v;
            make_atom<R>(P, key, i, A, p, v);
            W.pos[i] = p;
            W.vel[i] = v;
            W.term[i] = {R(0), R(0), R(0), R(0)};
        }
    } else {
        const unsigned char* rec = src == SRC_STOLEN ? B.pool + (size_t)S->slot * B.entry_bytes
                                                     : stack + (size_t)(S->top - 1) * B.entry_bytes;
        if (src == SRC_STOLEN) __threadfence();
        load_header<R>(S->ion, rec);
        load_window<R>(P, W, rec);
        __syncwarp();
        if (lane == 0) {
            if (src == SRC_STOLEN) {
                __threadfence();
                atomicExch(&B.pool_state[S->slot], (unsigned)POOL_EMPTY);
                atomicSub(&B.pool_ctl[1], 1u);
                if (B.splits) atomicAdd(&B.splits[REED_MAX_THR], 1ull);
            } else {
                S->top -= 1;
            }
        }
    }
    __syncwarp();
    return src;
}

// One clone of the track per cloning level passed (Sec. 2, Fig. "split"): a
// complete record to the pool while some CTA is idle, else to this CTA's
// stack.  S->ion holds the track's state; its level goes up by nc.  Returns
// the number of clones made (fewer than nc when the stack is full).
template <typename R, typename Head>
__device__ __noinline__ int push_clones(const DevParams& P, const DevBuf& B, Head* S, V4<R>* pos, V4<R>* vel,
                                        V4<R>* term, unsigned char* stack, int nc)
{
    const int lane = threadIdx.x & 31;
    for (int c = 0; c < nc; ++c) {
        int slot = -1;
        if (lane == 0 && B.pool && *(volatile unsigned*)&B.pool_ctl[0] > 0u) {
            atomicAdd(&B.pool_ctl[1], 1u);   // counted before the slot is visible
            slot = pool_claim(B, POOL_EMPTY, POOL_WRITING);
            if (slot < 0) atomicSub(&B.pool_ctl[1], 1u);
        }
        slot = __shfl_sync(0xffffffffu, slot, 0);
        const int top = S->top;
        if (slot < 0 && (top >= B.stack_depth || stack == nullptr)) {
            // the track still passes the levels (its depths stay in step with its
            // weight 2^-level), so the dropped clones' weight is lost from the
            // profile; the run reports REED_E_QUEUE_FULL
            if (lane == 0) {
                atomicOr(B.status, ERR_QUEUE);
                S->ion.level += nc - c;
            }
            __syncwarp();
            return c;
        }
        unsigned char* rec = slot >= 0 ? B.pool + (size_t)slot * B.entry_bytes : stack + (size_t)top * B.entry_bytes;
        if (lane == 0) {
            S->ion.level += 1;
            IonState<R> C = S->ion;
            C.id = clone_id(C.id, C.level);
            C.key = track_key(P.seed, C.id);
            *reinterpret_cast<IonState<R>*>(rec) = C;
            if (B.splits) atomicAdd(&B.splits[min(C.level, REED_MAX_THR) - 1], 1ull);
        }
        save_window<R, false>(P, pos, vel, term, rec);
        if (slot >= 0) __threadfence();
        __syncwarp();
        if (lane == 0) {
            if (slot >= 0) {
                atomicExch(&B.pool_state[slot], (unsigned)POOL_FULL);
                atomicAdd(&B.pool_ctl[2], 1u);
            } else {
                S->top = top + 1;
            }
        }
        __syncwarp();
    }
    return nc;
}

// Follow one track from its state in S->ion and W to its end (one warp);
// returns its end status, S->ion holds the final state.
template <typename R, bool ADJ, typename Head>
__device__ int follow_track(const DevParams& P, const DevBuf& B, const HotParams<R>& H, Head* S, IonWin<R>& W, int vt,
                            int src, unsigned char* stack, unsigned char* adjbase, int lane)
{
    IonRegs<R> I;
    unpack_ion<R>(I, S->ion, lane);
    const int nthr = S->nthr;
    const bool tracing = src == SRC_PRIMARY && S->pidx < P.trace_tracks;
    const long long pidx = S->pidx;
    regs_frame<R>(P, I, S->thr, nthr, lane);
    auto build = [&](const int Aold[3], bool shift, bool clear) {
        const R vm = build_ion_list<R>(P, B, S, W.pos, W.vel, W.term, W.list, W.hit, I.rel[0], I.rel[1], I.rel[2], I.A[0],
                                       I.A[1], I.A[2], Aold[0], Aold[1], Aold[2], I.level, shift, clear);
        W.nlist = S->need_count;
        W.nhit = S->nhit0;
        W.bx = I.rel[0];
        W.by = I.rel[1];
        W.bz = I.rel[2];
        return vm;
    };
    build(I.A, false, false);
    int nactive = S->active_count;
    {
        if (src == SRC_PRIMARY) {   // forces at the start
            R vm = R(0), pm = R(0);
            I.dt = R(0);
            ion_pair_pass<R, false>(P, H, W, I, R(0), vm, pm);
            ion_sums<R>(P, W, I, vt);
            if (ADJ) {   // checkpoint of the state before step 0
                pack_ion<R>(I, S->ion, lane);
                if (lane == 0) *reinterpret_cast<IonState<R>*>(adjbase) = S->ion;
                save_window<R, true>(P, W.pos, W.vel, W.term, adjbase);
                __syncwarp();
            }
        }
    }
    const long long steps0 = I.steps;
    const R skin2 = R((REED_ION_SKIN - 1e-3) * (REED_ION_SKIN - 1e-3));
    int status = 0;
    // work and clocks since the last flush, in 32 bits
    unsigned since = 0, pairs = 0, c_ion = 0, c_force = 0, t0 = (unsigned)clock();
    auto flush = [&]() {
        if (lane == 0) {
            S->cnt[ION_MOVED] += (unsigned long long)since * (unsigned)nactive;
            S->cnt[ION_PAIRS] += pairs;
            S->cnt[ION_PH_ION] += c_ion;
            S->cnt[ION_PH_FORCE] += c_force;
        }
        since = pairs = c_ion = c_force = 0;
    };
    for (;;) {
        int Aold[3];
        const bool on1 = I.rel[2] >= I.zsurf;
        const bool shift = regs_prologue<R>(P, H, I, Aold, S->thr, nthr, lane);
        const unsigned t1 = (unsigned)clock();
        c_ion += t1 - t0;
        const R hdt = R(0.5) * I.dt;
        ++since;
        const R ex = I.rel[0] - W.bx, ey = I.rel[1] - W.by, ez = I.rel[2] - W.bz;
        // (also taken when the position is not finite)
        const bool rebuild = shift || !(ex * ex + ey * ey + ez * ez < skin2);
        R vm = R(0), pm = R(0);
        // half kick and drift of the moving atoms, cutoff test; two entries
        // per lane at a time so that their loads overlap
        int nh = 0;
        for (int e0 = lane; e0 - lane < W.nlist; e0 += 64) {
            const bool on0 = e0 < W.nlist, onb = e0 + 32 < W.nlist;
            const int i0 = on0 ? W.list[e0] : 0, i1 = onb ? W.list[e0 + 32] : 0;
            const V4<R> p0 = W.pos[i0], v0 = W.vel[i0], f0 = W.term[i0];
            const V4<R> p1 = W.pos[i1], v1 = W.vel[i1], f1 = W.term[i1];
            bool h0 = false, h1 = false;
            if (on0) h0 = ion_move_atom<R>(H, W, I, i0, p0, v0, f0, hdt, !rebuild, vm);
            if (onb) h1 = ion_move_atom<R>(H, W, I, i1, p1, v1, f1, hdt, !rebuild, vm);
            if (!rebuild) {
                const unsigned b0 = __ballot_sync(0xffffffffu, h0), b1 = __ballot_sync(0xffffffffu, h1);
                const unsigned below = (1u << lane) - 1u;
                const int n0 = __popc(b0);
                if (h0) W.hit[nh + __popc(b0 & below)] = (uint16_t)i0;
                if (h1) W.hit[nh + n0 + __popc(b1 & below)] = (uint16_t)i1;
                nh += n0 + __popc(b1);
            }
        }
        __syncwarp();
        W.nhit = nh;
        if (rebuild) {
            flush();
            vm = build(Aold, shift, true);
            nactive = S->active_count;
            if (shift && lane == 0) S->cnt[ION_SHIFTS] += 1;
        } else if (since >= 4096u) {
            flush();
        }
        ion_pair_pass<R, true>(P, H, W, I, hdt, vm, pm);
        pairs += (unsigned)W.nhit;
        ion_sums<R>(P, W, I, vt);
        I.vmax2 = warp_max_pos(vm);
        I.pmax = H.de_max > R(0) ? warp_max_pos(pm) : R(0);
        t0 = (unsigned)clock();
        c_force += t0 - t1;
        // second half kick of the ion, end and cloning checks (see ion_step)
        const bool on2 = I.rel[2] >= I.zsurf;
        regs_kick<R>(H, I);
        I.acc += lane == 3 ? (double)I.dt : 0.0;
        I.steps += 1;
        const R E = R(0.5) * H.M1 * dist2(I.v[0], I.v[1], I.v[2]);
        const R far = I.rel[0] + I.rel[1] + I.rel[2];
        if (!(E >= H.e_stop) || !isfinite(E) || !isfinite(far) || (I.rel[2] < I.zback && I.v[2] < R(0)) ||
            I.steps >= P.step_cap) {
            if (!isfinite(E) || !isfinite(far)) status = REED_TRACK_FAILED;
            else if (E < H.e_stop) status = REED_TRACK_STOPPED;
            else if (I.rel[2] < I.zback && I.v[2] < R(0)) status = REED_TRACK_BACKSCATTERED;
            else status = REED_TRACK_TRUNCATED;
        }
        if (tracing && I.steps <= P.trace_steps) {
            const size_t o = (size_t)pidx * P.trace_steps + (size_t)(I.steps - 1);
            double* t8 = B.trace + 8 * o;
            if (lane < 4) t8[lane] = I.acc;
            if (lane == 0) {
                t8[4] = I.v[0]; t8[5] = I.v[1]; t8[6] = I.v[2]; t8[7] = I.dt;
                int* a3 = B.trace_anchor + 3 * o;
                a3[0] = I.A[0]; a3[1] = I.A[1]; a3[2] = I.A[2];
            }
        }
        if (ADJ) {
            // frozen quantities of this step; checkpoints every adj_every steps
            if (lane == 0) {
                StepRec<R>* ring = reinterpret_cast<StepRec<R>*>(adjbase + (size_t)P.adj_nck * B.entry_bytes);
                StepRec<R> sr;
                sr.dt = I.dt;
                sr.A[0] = I.A[0];
                sr.A[1] = I.A[1];
                sr.A[2] = I.A[2];
                sr.flags = (on1 ? 1 : 0) | (on2 ? 2 : 0) | (shift ? 4 : 0);
                ring[(I.steps - 1) % REED_STEP_RING] = sr;
            }
            if (!status && I.steps % P.adj_every == 0) {
                unsigned char* rec = adjbase + (size_t)((I.steps / P.adj_every) % P.adj_nck) * B.entry_bytes;
                pack_ion<R>(I, S->ion, lane);
                if (lane == 0) *reinterpret_cast<IonState<R>*>(rec) = S->ion;
                save_window<R, true>(P, W.pos, W.vel, W.term, rec);
                __syncwarp();
            }
        }
        if (status) break;
        bool check = I.rel[2] >= I.zthr;
        if (P.bulk && nthr > 0) {
            const R sx = R(I.A[0]) * H.a + I.rel[0], sy = R(I.A[1]) * H.a + I.rel[1], sz = R(I.A[2]) * H.a + I.rel[2];
            check = sx * sx + sy * sy + sz * sz >= I.zthr;
        }
        if (check) {
            // passed one (or more) cloning depths: count them on the FP64 depth
            const double z = regs_depth<R>(P, I);
            int nc = 0;
            while (I.level + nc < nthr && z >= S->thr[I.level + nc]) ++nc;
            if (nc) {
                pack_ion<R>(I, S->ion, lane);
                const int made = push_clones<R>(P, B, S, W.pos, W.vel, W.term, stack, nc);
                if (lane == 0) {
                    S->cnt[ION_CLONES] += (unsigned)made;
                    S->cnt[ION_DROPS] += (unsigned)(nc - made);
                }
                I.level = S->ion.level;
                regs_frame<R>(P, I, S->thr, nthr, lane);   // next cloning depth
            }
        }
    }
    flush();
    if (lane == 0) S->cnt[ION_STEPS] += (unsigned long long)(I.steps - steps0);
    pack_ion<R>(I, S->ion, lane);
    return status;
}

// The persistent kernel of the ion-target-only model: one track per CTA.
// Without the adjoint a CTA is one warp.  With it (ADJ) a CTA has vt threads:
// the first warp follows the track, all of them run the reverse pass of the
// truncated-segment adjoint.  (Where a block of threads follows a track, with the
// adjoint or without: reed_track_kernel.)
template <typename R, bool ADJ>
__global__ void __launch_bounds__(ADJ ? 256 : 32, (ADJ ? (sizeof(R) == 4 ? 2 : 1) : (sizeof(R) == 4 ? 16 : 10)))
    reed_ion_kernel(const __grid_constant__ DevParams P, const __grid_constant__ DevBuf B, const int vt)
{
    using Head = std::conditional_t<ADJ, TrackShared<R>, IonShared<R>>;
    extern __shared__ __align__(16) unsigned char smem[];
    Head* S = reinterpret_cast<Head*>(smem);
    IonWin<R> W(smem, IonLayout<R, ADJ>::head_bytes(), P.na, ADJ);
    const HotParams<R>& H = hot<R>(P);
    const int tid = threadIdx.x, lane = tid & 31;
    unsigned char* adjbase = (ADJ && B.adj) ? B.adj + (size_t)blockIdx.x * B.adj_stride : nullptr;
    unsigned char* stack = B.stacks ? B.stacks + (size_t)blockIdx.x * B.stack_stride : nullptr;
    long long t_mark = clock64();
    if (tid == 0) {
        S->top = 0;
        S->was_busy = 0;
        for (int c = 0; c < ION_NCOUNT; ++c) S->cnt[c] = 0;
    }
    if (ADJ) __syncthreads();
    else __syncwarp();
    for (;;) {
        if (!ADJ || tid < 32) {
            const int src = acquire_track<R>(P, B, S, W, stack, lane);
            if (src != SRC_NONE) {
                if (lane == 0) {
                    if (src == SRC_PRIMARY) S->cnt[ION_PRIM] += 1;
                    S->cnt[ION_PH_ADMIN] += (unsigned long long)(clock64() - t_mark);
                }
                const int status = follow_track<R, ADJ>(P, B, H, S, W, vt, src, stack, adjbase, lane);
                t_mark = clock64();
                if (B.damage) {
                    const int A[3] = {S->ion.A[0], S->ion.A[1], S->ion.A[2]};
                    const double wgt = ldexp(1.0, -S->ion.level);
                    for (int i = lane; i < P.na; i += 32) {
                        const V4<R> p = W.pos[i];
                        if (is_active(p)) deposit_damage<R>(P, B, p, W.vel[i], A, wgt);
                    }
                }
                if (lane == 0) {
                    S->cnt[ION_TRACKS] += 1;
                    if (status == REED_TRACK_FAILED) {
                        S->cnt[ION_FAILS] += 1;
                        atomicOr(B.status, ERR_NONFINITE);
                    }
                    const long long k = finish_track<R>(P, B, S->ion, status);
                    if constexpr (ADJ) {
                        S->rec_index = k;
                        S->status = status;
                    }
                }
                __syncwarp();
            }
        }
        if (ADJ) __syncthreads();
        const int src = S->src;
        if (!ADJ) __syncwarp();   // (lane 0 goes on to write the next track's; an adjoint run ends on a barrier)
        if (src == SRC_NONE) break;
        if constexpr (ADJ) {
            Win<R, REED_TT_NONE> WA(smem, P.na, 0, 1);
            adjoint_gradient<R>(P, B, H, WA, adjbase);
            __syncthreads();
        }
    }
    if (tid == 0) {
        S->cnt[ION_PH_ADMIN] += (unsigned long long)(clock64() - t_mark);
        constexpr int to[ION_NCOUNT] = {C_PRIMARIES, C_CLONES, C_TRACKS, C_STEPS, C_PAIRS, C_SHIFTS, C_DROPPED, C_FAILED,
                                        C_MOVED, C_PHASE0 + PH_ION, C_PHASE0 + PH_FORCE, C_PHASE0 + PH_ADMIN};
        for (int c = 0; c < ION_NCOUNT; ++c) atomicAdd(&B.counters[to[c]], S->cnt[c]);
    }
}
