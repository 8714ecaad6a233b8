// lbfe_passes.cu -- the time step as three passes over the lattice inside one
// persistent kernel, several steps per launch:
//
//   pass M   densities, momentum and stress scalars of every cell (stage M);
//   pass X   forces, velocity, collision and push streaming (stages F and X);
//   pass U   the FENE-P update of the conformation (stage U)
// (the stages are described in lbfe_step.cuh; every expression is the one of
// the tile kernels, so that the fields are theirs bit for bit).
//
// Why besides the tile kernels.  Those read each population once, but a block
// marches a 32-wide column tile plane by plane (about 3.2 us a plane whatever
// it holds), recomputes the moments of the cells around it and wants rows of
// 16-byte multiples.  The passes know no tiles: cells are taken in memory order,
// in runs of 256, whatever the extents, nothing is computed twice, and a
// lattice of few columns still fills the GPU.  They pay with the populations'
// second read (the L2 serves part of it), 40 bytes a cell of scratch and more
// instructions.  Measured in FP32, tile kernel -> passes, us per step: 32^3
// 37 -> 15, 64^3 38 -> 32, 141 x 75 x 53 104 -> 62, sixteen 320 x 44 x 40
// 997 -> 991; 192 x 96 x 80 144 -> 162 (the tile kernel stays), in calls of
// twenty steps.
// Which of the two a handle runs is decided in lbfe_capi.cu (takes_passes).
//
// Work.  A slot is one pass over up to R x 256 cells.  Slots are numbered so
// that passes M, X and U of the lattice follow one another at fixed distances
// (lag_x, lag_u), step after step, and are taken in that order from a counter
// (one block per SM, two teams per block).  A slot waits until the planes it
// reads have been finished by the pass before (counters per plane and pass);
// it only ever waits for slots with smaller numbers.  Every slot comes from the
// counter, the first one of a team too, so that those have all been taken by
// running teams, and the smallest unfinished one waits for nothing: the waits
// end however many blocks are resident, also beside other kernels.  They are
// bounded all the same.
// What overwrites what: X(t+1) writes the populations read by M(t) and X(t),
// U(t+1) the conformation read by X(t) and U(t), M(t+1) the scratch read by
// X(t); each of these is implied by the waits, which cover the planes on
// either side.
//
// A team is a scheduling warp and eight computing warps.  The scheduling warp
// takes slots, waits for their inputs and starts the copies: one TMA box holds
// a run's 38 populations, two runs are in flight, so the collision's loads
// hide behind the stencils' and behind the wait of the next slot.  With the
// populations in registers (38 ordinary loads ahead of the stencil) the
// 192 x 96 x 80 step took 186 us, with staging 166, with the scheduling warp
// 160, with the L2 hints of the copies 154 (with packed stencil sums; 160 with
// the tile kernels' sums, which keep the bits, and ONE).
// Bound by latency at sixteen computing warps of 104 or 112 registers (issue
// slots 38 % busy) and, on large lattices, DRAM (about 530 bytes a cell).
#include <type_traits>

#include "lbfe_step.cuh"

namespace lbfe {

namespace {

constexpr int kRun = 256;            // cells of a run, computing threads of a team
constexpr int kTeams = 2;
constexpr int kPassThreads = kTeams * kRun + 128;   // and a warpgroup with the scheduling warps
constexpr int kMaxRuns = 4;          // most runs of a slot (8: slower, the slots in flight outgrow the L2)
constexpr int kPassSteps = 16;       // most steps of a launch

// Per-instance descriptor (kernel parameter space).
struct PassInst {
    const void *f[2];
    const CUtensorMap *runs[2];      // populations as [38][S], box 256 x 38
    float *C[2];
    float2 *dens[2];
    float2 *rho, *pi;                // scratch: densities, stress scalars (a f, a)
    float *j, *u;                    // scratch [3][S]: momentum, velocity
    unsigned *cnt;                   // finished cells [3][Lz] by pass and plane, then their value at launch
    unsigned *status, *step_ctr;
    float G, Uw, nu_A, nu_B, pi_coef, L2, inv_tauP, gx, gy, gz, rho0A, rho0B;
    u32 S, N, LxLy;
    u32 mul_p, mul_x;                // reciprocals of LxLy and Lx (div_by)
    unsigned short Lx, Ly, Lz;
    unsigned char sh_p, sh_x;
    signed char visc_comp;
};

struct PassArgs {
    int n, steps, parity;            // parity: ping-pong index of the state the first step reads
    int R, items;                    // runs of a slot; slots of one pass
    int period, lag_x, lag_u;        // distance of two steps; of the passes of a step
    int slots;
    int lost;                        // test hook: pass M is not counted
    unsigned *status;
    unsigned *work;                  // [0] slots taken, [1] finished teams, kGaveUp; zero between launches
    int item_off[kStepMaxInst + 1];  // first slot of each instance
    PassInst inst[kStepMaxInst];
};
static_assert(sizeof(PassArgs) < 32000, "kernel parameter space");
constexpr unsigned kGaveUp = 1u << 31;   // a wait of the launch has expired

// n / d by the reciprocal of fast_div.
__device__ __forceinline__ u32 div_by(u32 n, u32 mul, u32 sh) {
    const u32 t = __umulhi(mul, n);
    return (t + ((n - t) >> (sh >> 7))) >> (sh & 31u);
}

__device__ __forceinline__ unsigned ld_relaxed(const unsigned *p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// Report an expired wait to the host and to the launch's other waits.
__device__ __forceinline__ void give_up(const PassArgs &A) {
    atomicOr(A.status, kFlagTimeout);
    atomicOr(A.work + 1, kGaveUp);
}

// Wait until *p has reached target; false once a wait of the launch expired,
// here or anywhere.
__device__ __forceinline__ bool wait_count(const unsigned *p, unsigned target, const PassArgs &A) {
    unsigned long long t0 = 0;
    for (u32 it = 0; it < kWaitRounds; ++it) {
        if ((int)(ld_relaxed(p) - target) >= 0) return true;
        if ((it & 255u) == 255u) {
            if (ld_relaxed(A.work + 1) & kGaveUp) return false;
            const unsigned long long now = global_ns();
            if (t0 == 0)
                t0 = now;
            else if (now - t0 > kWaitNs)
                break;
        }
    }
    give_up(A);
    return false;
}

__device__ __forceinline__ void raise(unsigned *status, const PassInst &I) {
    atomicOr(status, kFlagDiverged);
    if (I.status) atomicOr(I.status, kFlagDiverged);
}

template <typename T>
__device__ __forceinline__ float2 offsets_at(const PassInst &I, int b, u32 n) {
    if (!Store<T>::offset) return bc(0.f);
    if (I.dens[0]) return __ldcg(I.dens[b ^ 1] + n);
    return make_float2(I.rho0A, I.rho0B);
}

// What other blocks wrote in this launch: cached loads, never read-only ones.
template <typename V>
__device__ __forceinline__ V ldc(const V *p) {
    return __ldca(p);
}

// ---------------------------------------------------------------- pass M
// Cell n (st: its column of the staged run; on: inside the slot).  wait()
// returns once the run is there.
template <typename T, typename Wait>
__device__ __forceinline__ void pass_m(const PassInst &I, int b, u32 n, bool on, const T *st, Wait &&wait) {
    const float *C = I.C[b];
    const u32 S = I.S;
    const float2 o = offsets_at<T>(I, b, n);
    const float c0 = __ldcg(C + n), c1 = __ldcg(C + (S + n)), c2 = __ldcg(C + (2 * S + n));
    wait();
    float2 ab[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) {
        ab[i].x = Store<T>::ld_plain(st + i * kRun);
        ab[i].y = Store<T>::ld_plain(st + (Q + i) * kRun);
        if (Store<T>::offset) ab[i] = fma2(bc(wq(i)), o, ab[i]);
    }
    float2 r = ab[0];
#pragma unroll
    for (int i = 1; i < Q; ++i) r = add2(r, ab[i]);
    float2 jx = bc(0.f), jy = jx, jz = jx;
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
        const float2 d = sub2(ab[i], ab[i + 1]);
        if (cx(i)) jx = cx(i) > 0 ? add2(jx, d) : sub2(jx, d);
        if (cy(i)) jy = cy(i) > 0 ? add2(jy, d) : sub2(jy, d);
        if (cz(i)) jz = cz(i) > 0 ? add2(jz, d) : sub2(jz, d);
    }
    if (!on) return;
    I.rho[n] = r;
    I.j[n] = jx.x + jx.y;
    I.j[S + n] = jy.x + jy.y;
    I.j[2 * S + n] = jz.x + jz.y;
    if (I.visc_comp >= 0) {
        const float a = I.pi_coef * (I.visc_comp == 0 ? r.x : r.y) / (r.x + r.y);
        const float fp = peterlin(I.L2, c0, c1, c2);
        I.pi[n] = make_float2(a * fp, a);
    }
}

// Offsets of a cell's neighbours: periodic in x and y, the wall layer itself
// beyond a wall.
struct Place {
    int xp, xm, yp, ym, zp, zm;
    u32 x, y, z;
};

__device__ __forceinline__ Place place_of(const PassInst &I, u32 n) {
    Place P;
    const int Lx = I.Lx, LxLy = (int)I.LxLy;
    P.z = div_by(n, I.mul_p, I.sh_p);
    const u32 r = n - P.z * I.LxLy;
    P.y = div_by(r, I.mul_x, I.sh_x);
    P.x = r - P.y * (u32)Lx;
    P.xp = (int)P.x == Lx - 1 ? 1 - Lx : 1;
    P.xm = P.x == 0 ? Lx - 1 : -1;
    P.yp = (int)P.y == I.Ly - 1 ? Lx - LxLy : Lx;
    P.ym = P.y == 0 ? LxLy - Lx : -Lx;
    P.zp = (int)P.z == I.Lz - 1 ? 0 : LxLy;
    P.zm = P.z == 0 ? 0 : -LxLy;
    return P;
}

__device__ __forceinline__ int off_of(const Place &P, int i) {
    return (cx(i) > 0 ? P.xp : (cx(i) < 0 ? P.xm : 0)) + (cy(i) > 0 ? P.yp : (cy(i) < 0 ? P.ym : 0)) +
           (cz(i) > 0 ? P.zp : (cz(i) < 0 ? P.zm : 0));
}

// ---------------------------------------------------------------- pass X
template <typename T, typename Wait>
__device__ __forceinline__ void pass_x(const PassInst &I, int b, u32 n, bool on, unsigned seed, unsigned *status,
                                       const T *st, Wait &&wait) {
    T *fo = (T *)I.f[b ^ 1];
    const float *C = I.C[b];
    const u32 S = I.S;
    const Place P = place_of(I, n);
    const int m = (int)n;
    const float2 o = offsets_at<T>(I, b, n);
    const float2 *rho = I.rho;
    const float2 r0 = ldc(rho + n);
    float2 nb[Q];
#pragma unroll
    for (int i = 1; i < Q; ++i) nb[i] = ldc(rho + m + off_of(P, i));
    const float j[3] = {ldc(I.j + n), ldc(I.j + S + n), ldc(I.j + 2 * S + n)};
    const bool visc = I.visc_comp >= 0;
    float2 Ax, Bx, Ay, By, Az, Bz;
    float xp[3], xm[3], yp[3], ym[3], zp[3], zm[3];
    if (visc) {
        const float2 *pi = I.pi;
        const float *c0 = C, *c1 = C + S, *c2 = C + 2 * S, *c3 = C + 3 * S, *c4 = C + 4 * S, *c5 = C + 5 * S;
        Ax = ldc(pi + m + P.xp); Bx = ldc(pi + m + P.xm);
        Ay = ldc(pi + m + P.yp); By = ldc(pi + m + P.ym);
        Az = ldc(pi + m + P.zp); Bz = ldc(pi + m + P.zm);
        // rows of C that the divergence along each axis takes
        xp[0] = ldc(c0 + m + P.xp); xm[0] = ldc(c0 + m + P.xm); xp[1] = ldc(c3 + m + P.xp); xm[1] = ldc(c3 + m + P.xm);
        xp[2] = ldc(c4 + m + P.xp); xm[2] = ldc(c4 + m + P.xm);
        yp[0] = ldc(c3 + m + P.yp); ym[0] = ldc(c3 + m + P.ym); yp[1] = ldc(c1 + m + P.yp); ym[1] = ldc(c1 + m + P.ym);
        yp[2] = ldc(c5 + m + P.yp); ym[2] = ldc(c5 + m + P.ym);
        zp[0] = ldc(c4 + m + P.zp); zm[0] = ldc(c4 + m + P.zm); zp[1] = ldc(c5 + m + P.zp); zm[1] = ldc(c5 + m + P.zm);
        zp[2] = ldc(c2 + m + P.zp); zm[2] = ldc(c2 + m + P.zm);
    }
    // every load is on its way before the first use (the compiler would keep
    // a few in flight otherwise)
    __syncwarp();
    const float rA = r0.x, rB = r0.y;
    float sA[3] = {0.f, 0.f, 0.f}, sB[3] = {0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
        const float dA = nb[i].x - nb[i + 1].x, dB = nb[i].y - nb[i + 1].y, w = wq(i);
        if (cx(i)) { sA[0] += cx(i) * w * dB; sB[0] += cx(i) * w * dA; }
        if (cy(i)) { sA[1] += cy(i) * w * dB; sB[1] += cy(i) * w * dA; }
        if (cz(i)) { sA[2] += cz(i) * w * dB; sB[2] += cz(i) * w * dA; }
    }
    float FP[3] = {0.f, 0.f, 0.f};
    if (visc) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            float gxd = Ax.x * xp[a] - Bx.x * xm[a];
            float gyd = Ay.x * yp[a] - By.x * ym[a];
            float gzd = Az.x * zp[a] - Bz.x * zm[a];
            if (a == 0) gxd -= Ax.y - Bx.y;
            if (a == 1) gyd -= Ay.y - By.y;
            if (a == 2) gzd -= Az.y - Bz.y;
            FP[a] = 0.5f * (gxd + gyd + gzd);
        }
    }
    const float g[3] = {I.gx, I.gy, I.gz};
    const float inv = 1.0f / (rA + rB);
    float2 F[3];
    float u[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float FA = -I.G * rA * sA[a] + (rA * inv) * FP[a] + rA * g[a];
        const float FB = -I.G * rB * sB[a] + (rB * inv) * FP[a] + rB * g[a];
        u[a] = (j[a] + 0.5f * (FA + FB)) * inv;
        F[a] = make_float2(FA, FB);
        if (on) I.u[a * S + n] = u[a];
    }
    const float rt = rA + rB;
    if (on && (!(rt > 0.f) || u[0] != u[0] || u[1] != u[1] || u[2] != u[2])) raise(status, I);
    // omega = 1 / (3 nu + 1/2), nu = (rho_A nu_A + rho_B nu_B) / rho
    const float om = rt / (3.0f * (rA * I.nu_A + rB * I.nu_B) + 0.5f * rt);
    wait();
    if (!on) return;
    auto pop = [&](int i) {
        float2 v = make_float2(Store<T>::ld_plain(st + i * kRun), Store<T>::ld_plain(st + (Q + i) * kRun));
        if (Store<T>::offset) v = fma2(bc(wq(i)), o, v);
        return v;
    };
    const bool track = I.dens[0] != nullptr;
    const bool bottom = P.z == 0, top = (int)P.z == I.Lz - 1;
    auto push = [&](int i, float2 v) {
        int dir = i, dst = m + off_of(P, i);
        float2 od = nb[i];           // densities at the destination
        if ((cz(i) < 0 && bottom) || (cz(i) > 0 && top)) {
            v = fma2(bc(-6.f * wq(i) * (float)cx(i) * (cz(i) < 0 ? -I.Uw : I.Uw)), r0, v);
            dir = opp(i);
            dst = m;
            od = r0;
        }
        if (Store<T>::offset) v = fma2(bc(-wq(i)), track ? od : make_float2(I.rho0A, I.rho0B), v);
        const unsigned r = Store<T>::sround ? sround_bits((u32)dst, dir, seed) : 0u;
        Store<T>::st_sr(fo + (u32)(dir * S + (u32)dst), v.x, r);
        Store<T>::st_sr(fo + (u32)((Q + dir) * S + (u32)dst), v.y, r >> 16);
    };
    // the packed BGK + Guo collision of collide_push_ab
    const float omc = 1.0f - om, pref = 1.0f - 0.5f * om;
    const float uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
    const float2 u2[3] = {bc(u[0]), bc(u[1]), bc(u[2])};
    const float2 uF = fma2(u2[2], F[2], fma2(u2[1], F[1], mul2(u2[0], F[0])));
    const float2 E = fma2(bc(-3.f * pref), uF, mul2(bc(om * (1.f - 1.5f * uu)), r0));
    const float2 omc2 = bc(omc);
    {
        float2 v = fma2(omc2, pop(0), mul2(bc(wq(0)), E));
        if (Store<T>::offset) v = fma2(bc(-wq(0)), track ? r0 : make_float2(I.rho0A, I.rho0B), v);
        const unsigned r = Store<T>::sround ? sround_bits(n, 0, seed) : 0u;
        Store<T>::st_sr(fo + n, v.x, r);
        Store<T>::st_sr(fo + (u32)(Q * S + n), v.y, r >> 16);
    }
    float2 Ew[2], a1w[2], b1w[2], a2w[2], b2w[2];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
        const float w = wq(c == 0 ? 1 : 7);
        Ew[c] = mul2(bc(w), E);
        a1w[c] = mul2(bc(4.5f * om * w), r0);
        b1w[c] = bc(9.f * pref * w);
        a2w[c] = mul2(bc(3.f * om * w), r0);
        b2w[c] = bc(3.f * pref * w);
    }
#pragma unroll
    for (int i = 1; i < Q; i += 2) {
        const int c = i <= 6 ? 0 : 1;
        float2 cu = bc(0.f), cF = cu;
        bool first = true;
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int ca = a == 0 ? cx(i) : (a == 1 ? cy(i) : cz(i));
            if (!ca) continue;
            if (first) {             // +1 in every odd direction
                cu = u2[a];
                cF = F[a];
                first = false;
            } else {
                cu = ca > 0 ? add2(cu, u2[a]) : sub2(cu, u2[a]);
                cF = ca > 0 ? add2(cF, F[a]) : sub2(cF, F[a]);
            }
        }
        const float2 sym = fma2(cu, fma2(a1w[c], cu, mul2(b1w[c], cF)), Ew[c]);
        const float2 anti = fma2(a2w[c], cu, mul2(b2w[c], cF));
        const float2 fi = pop(i), fj = pop(i + 1);
        push(i, fma2(omc2, fi, add2(sym, anti)));
        push(i + 1, fma2(omc2, fj, sub2(sym, anti)));
    }
    // this step's densities: the offsets of the state just written
    if (Store<T>::offset && track) I.dens[b][n] = r0;
}

// ---------------------------------------------------------------- pass U
template <bool ADV2>
__device__ __forceinline__ void pass_u(const PassInst &I, int b, u32 n, bool on, unsigned *status) {
    const float *C = I.C[b];
    float *Cn = I.C[b ^ 1];
    const u32 S = I.S;
    const int m = (int)n;
    const Place P = place_of(I, n);
    const float Uw = I.Uw;
    float u0[3], uxp[3], uxm[3], uyp[3], uym[3], uzp[3], uzm[3], c[6];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const float *u = I.u + a * S;
        u0[a] = ldc(u + m);
        uxp[a] = ldc(u + m + P.xp); uxm[a] = ldc(u + m + P.xm);
        uyp[a] = ldc(u + m + P.yp); uym[a] = ldc(u + m + P.ym);
        uzp[a] = ldc(u + m + P.zp); uzm[a] = ldc(u + m + P.zm);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) c[k] = ldc(C + k * S + n);
    __syncwarp();
    const bool px = u0[0] > 0.f, py = u0[1] > 0.f, pz = u0[2] > 0.f;
    const float sx = px ? u0[0] : -u0[0], sy = py ? u0[1] : -u0[1], sz = pz ? u0[2] : -u0[2];
    const int ox = px ? P.xm : P.xp, oy = py ? P.ym : P.yp, oz = pz ? P.zm : P.zp;
    float adv[6];
    if constexpr (!ADV2) {
        float cx_[6], cy_[6], cz_[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const float *Ck = C + k * S;
            cx_[k] = ldc(Ck + m + ox);
            cy_[k] = ldc(Ck + m + oy);
            cz_[k] = ldc(Ck + m + oz);
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 6; ++k) adv[k] = sx * (c[k] - cx_[k]) + sy * (c[k] - cy_[k]) + sz * (c[k] - cz_[k]);
    } else {
        // the second neighbours upwind and the first ones downwind
        const int x = (int)P.x, y = (int)P.y, z = (int)P.z, Lz = I.Lz;
        const int oxx = wrapg(px ? x - 2 : x + 2, I.Lx) - x, oyy = (wrapg(py ? y - 2 : y + 2, I.Ly) - y) * I.Lx,
                  ozz = (min(max(pz ? z - 2 : z + 2, 0), Lz - 1) - z) * (int)I.LxLy;
        const int bx = px ? P.xp : P.xm, by = py ? P.yp : P.ym, bz = pz ? P.zp : P.zm;
        auto lim = [](float c0, float a, float aa, float d) {
            return (c0 - a) + 0.5f * (minmodf(d - c0, c0 - a) - minmodf(c0 - a, a - aa));
        };
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            const float *Ck = C + k * S;
            adv[k] = sx * lim(c[k], ldc(Ck + m + ox), ldc(Ck + m + oxx), ldc(Ck + m + bx)) +
                     sy * lim(c[k], ldc(Ck + m + oy), ldc(Ck + m + oyy), ldc(Ck + m + by)) +
                     sz * lim(c[k], ldc(Ck + m + oz), ldc(Ck + m + ozz), ldc(Ck + m + bz));
        }
    }
    if (!on) return;
    float Gr[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float uwb = k == 0 ? -Uw : 0.f, uwt = k == 0 ? Uw : 0.f;
        const float up = ((int)P.z == I.Lz - 1) ? 2.f * uwt - u0[k] : uzp[k];
        const float dn = (P.z == 0) ? 2.f * uwb - u0[k] : uzm[k];
        Gr[0][k] = 0.5f * (uxp[k] - uxm[k]);
        Gr[1][k] = 0.5f * (uyp[k] - uym[k]);
        Gr[2][k] = 0.5f * (up - dn);
    }
    const float Cm[3][3] = {{c[0], c[3], c[4]}, {c[3], c[1], c[5]}, {c[4], c[5], c[2]}};
    const float fp = peterlin(I.L2, c[0], c[1], c[2]);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
        const int a = k < 3 ? k : (k == 5 ? 1 : 0);
        const int d = k < 3 ? k : (k == 3 ? 1 : 2);
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < 3; ++q) s += Cm[a][q] * Gr[q][d] + Gr[q][a] * Cm[q][d];
        const float relax = (fp * c[k] - (k < 3 ? 1.f : 0.f)) * I.inv_tauP;
        Cn[k * S + n] = c[k] + (-adv[k] + s - relax);
    }
    if (!(c[0] + c[1] + c[2] < I.L2)) raise(status, I);
}

// ---------------------------------------------------------------- the kernel
// Registers of the scheduling warpgroup and of the computing threads; the
// block is launched with 96 each.
template <typename T> constexpr int kAuxRegs = sizeof(T) == 4 ? 64 : 32;
template <typename T> constexpr int kMainRegs = sizeof(T) == 4 ? 104 : 112;
static_assert(128 * kAuxRegs<float> + kTeams * kRun * kMainRegs<float> <= 96 * kPassThreads, "register split");
static_assert(128 * kAuxRegs<__half> + kTeams * kRun * kMainRegs<__half> <= 96 * kPassThreads, "register split");

template <int N, bool INC>
__device__ __forceinline__ void set_regs() {
    if constexpr (INC)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
    else
        asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// A slot as a team works on it: one pass over the cells [c0, c1) of instance k.
struct Job {
    int pass, k, step;               // pass 3: no more
    u32 c0, c1;
};
constexpr int kPassEnd = 3;

template <typename T>
constexpr int pass_smem() {
    return kTeams * 2 * 2 * Q * kRun * (int)sizeof(T) + 128;
}

// ONE: a launch of one instance, whose descriptor's address is then a constant
// (base addresses in uniform registers: 192 x 96 x 80 164 -> 160 us in FP32,
// 180 -> 165 in FP16).
template <typename T, bool ADV2, bool ONE>
__global__ void __launch_bounds__(kPassThreads, 1) k_passes(const __grid_constant__ PassArgs A) {
    __shared__ Job t_job[kTeams][2], t_cur[kTeams];   // handed over; worked on
    // per team, two of each: run copied, run read, job known, job read
    __shared__ __align__(8) unsigned long long t_full[kTeams][2], t_free[kTeams][2], t_jfull[kTeams][2],
        t_jfree[kTeams][2];
    __shared__ int t_how[kTeams];
    constexpr u32 kStage = (u32)(2 * Q * kRun * sizeof(T));
    static_assert(kStage % 128 == 0, "copy alignment");
    const bool computing = threadIdx.x < kTeams * kRun;
    const int team = computing ? (int)threadIdx.x / kRun : ((int)threadIdx.x - kTeams * kRun) / 32;
    // one instruction for all warps of the last warpgroup, also those that only fill it
    if (!computing) set_regs<kAuxRegs<T>, false>();
    if (team >= kTeams) {
        __syncthreads();
        return;
    }
    const int t = computing ? (int)threadIdx.x % kRun : (int)threadIdx.x & 31;
    const u32 sbase = smem_addr(lbfe_smem4), stage_addr = ((sbase + 127u) & ~127u) + team * 2 * kStage;
    const char *stage0 = reinterpret_cast<const char *>(lbfe_smem4) + (stage_addr - sbase);
    Job *s_job = t_job[team];
    const u32 full = smem_addr(t_full[team]), freeb = smem_addr(t_free[team]), jfull = smem_addr(t_jfull[team]),
              jfree = smem_addr(t_jfree[team]);
    if (computing && t == 0) {
        for (int q = 0; q < 2; ++q) {
            mbar_init(full + 8 * q);
            mbar_init_count(freeb + 8 * q, kRun / 32);
            mbar_init(jfull + 8 * q);
            mbar_init(jfree + 8 * q);
        }
    }
    const u32 cells = (u32)(kRun * A.R);
    bool expired = false;
    u32 runs = 0, jobs = 0;          // runs staged, jobs taken so far

    if (!computing) {
        // ---- scheduling warp
        __syncthreads();
        // what pass M reads stays in the L2 for pass X, which reads it last
        unsigned long long keep, drop;
        asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(keep));
        asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(drop));
        auto take = [&]() {
            int next = A.slots;
            if (t == 0 && !expired) next = (int)atomicAdd(A.work, 1u);
            return __shfl_sync(0xffffffffu, next, 0);
        };
        // the place of the next job, once its last one has been read
        auto job_slot = [&]() { return jobs < 2 || mbar_wait(jfree + 8 * (jobs & 1), ((jobs >> 1) - 1) & 1u); };
        // The warp stops at its first expired wait: a job or a copy handed over
        // without that wait would overwrite one that is still being read.  runs and
        // jobs (lane 0) are what was handed over.
        for (int slot = take(); slot < A.slots; slot = take()) {
            const int pass = slot % 3;
            const int q = slot / 3 - (pass == 0 ? 0 : (pass == 1 ? A.lag_x : A.lag_u));
            const int step = q < 0 ? -1 : q / A.period;
            const int item = q < 0 ? 0 : q - step * A.period;
            if (step >= 0 && step < A.steps && item < A.items) {
                int k = 0;
                for (int hi = A.n - 1; k < hi;) {
                    const int mid = (k + hi + 1) >> 1;
                    if (A.item_off[mid] <= item) k = mid; else hi = mid - 1;
                }
                const PassInst &I = A.inst[ONE ? 0 : k];
                const int Lz = I.Lz;
                const u32 c0 = (u32)(item - A.item_off[k]) * cells, c1 = min(c0 + cells, I.N);
                // the pass before on the slot's planes and the ones beside them;
                // from the second step on also the passes whose inputs are
                // overwritten here
                if (pass > 0 || step > 0) {
                    const int zl = max((int)div_by(c0, I.mul_p, I.sh_p) - 1, 0);
                    const int zh = min((int)div_by(c1 - 1, I.mul_p, I.sh_p) + 1, Lz - 1);
                    const unsigned prev = ld_relaxed(I.cnt + 3 * Lz) + (unsigned)step * I.LxLy, now = prev + I.LxLy;
                    for (int z = zl + t; z <= zh && !expired; z += 32) {
                        bool ok = true;
                        if (pass == 1) ok = wait_count(I.cnt + z, now, A);
                        if (pass == 2 || (pass == 0 && ok)) ok = wait_count(I.cnt + Lz + z, pass == 2 ? now : prev, A);
                        if (pass < 2 && ok && step > 0) ok = wait_count(I.cnt + 2 * Lz + z, prev, A);
                        if (!ok) expired = true;
                    }
                    __threadfence();
                    expired = __any_sync(0xffffffffu, expired);
                }
                if (t == 0 && !expired && !job_slot()) expired = true;
                if (t == 0 && !expired) {
                    const int e = jobs & 1;
                    s_job[e] = Job{pass, k, step, c0, c1};
                    mbar_arrive(jfull + 8 * e);
                    ++jobs;
                    if (pass < 2) {
                        const CUtensorMap *map = I.runs[(A.parity + step) & 1];
                        asm volatile("fence.proxy.async;" ::: "memory");
                        for (u32 c = c0; c < c1; c += kRun) {
                            const int sg = runs & 1;
                            if (runs >= 2 && !mbar_wait(freeb + 8 * sg, ((runs >> 1) - 1) & 1u)) {
                                expired = true;
                                break;
                            }
                            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                            mbar_expect(full + 8 * sg, kStage);
                            asm volatile(
                                "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
                                ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(stage_addr + sg * kStage),
                                "l"(reinterpret_cast<unsigned long long>(map)), "r"((int)c), "r"(0),
                                "r"(full + 8 * sg), "l"(pass == 0 ? keep : drop)
                                : "memory");
                            ++runs;
                        }
                    }
                }
            }
        }
        if (t == 0) {
            // copies may still be in flight where a wait expired, here or in the computing
            // warps: the last one issued to each stage is waited for, bounded, before the
            // block's shared memory goes (at once where the computing warps have seen it)
            for (u32 q = 1; q <= 2 && q <= runs; ++q)
                if (!mbar_wait(full + 8 * ((runs - q) & 1), ((runs - q) >> 1) & 1u)) expired = true;
            if (expired) give_up(A);
            // the end is the last that the team hears of this warp
            if (job_slot()) {
                s_job[jobs & 1].pass = kPassEnd;
                mbar_arrive(jfull + 8 * (jobs & 1));
            }
        }
        return;
    }

    // ---- computing warps
    set_regs<kMainRegs<T>, true>();
    __syncthreads();
    auto team_barrier = [&]() { asm volatile("bar.sync %0, 256;" ::"r"(1 + team) : "memory"); };
    for (;; ++jobs) {
        // one thread takes the job, so that the team agrees on it (and on its end)
        // whatever the waits do; the scheduling warp's own waits come first, and have
        // all ended, with the warp, before this one expires
        if (t == 0) {
            const int e = jobs & 1;
            bool known = false;
            for (int tries = 0; tries < 16 && !known; ++tries) known = mbar_wait(jfull + 8 * e, (jobs >> 1) & 1u);
            if (known) {
                t_cur[team] = s_job[e];
                mbar_arrive(jfree + 8 * e);
            } else {
                t_cur[team].pass = kPassEnd;
                expired = true;
            }
        }
        team_barrier();
        const Job J = t_cur[team];
        const int pass = J.pass, b = (A.parity + J.step) & 1;
        if (pass == kPassEnd) break;
        const PassInst &I = A.inst[ONE ? 0 : J.k];
        const u32 c0 = J.c0, c1 = J.c1;
        if (pass < 2) {
            unsigned seed = 0;
            if (Store<T>::sround && I.step_ctr) seed = __ldcg(I.step_ctr + A.parity) + (unsigned)J.step;
            for (u32 c = c0; c < c1; c += kRun, ++runs) {
                const int sg = runs & 1;
                const u32 n = c + t;
                const T *st = reinterpret_cast<const T *>(stage0 + sg * kStage) + t;
                auto wait = [&]() {
                    if (!expired && !mbar_wait(full + 8 * sg, (runs >> 1) & 1u)) expired = true;
                    __syncwarp();
                };
                if (pass == 0)
                    pass_m<T>(I, b, min(n, c1 - 1), n < c1, st, wait);
                else
                    pass_x<T>(I, b, min(n, c1 - 1), n < c1, seed, A.status, st, wait);
                __syncwarp();
                // a stage whose copy was not seen to arrive is never handed back: the
                // scheduling warp's wait for it expires and it copies no more
                if ((t & 31) == 0 && !expired) mbar_arrive(freeb + 8 * sg);
            }
        } else {
            for (u32 c = c0; c < c1; c += kRun) pass_u<ADV2>(I, b, min(c + t, c1 - 1), c + t < c1, A.status);
        }
        team_barrier();
        // publish the slot's cells, plane by plane
        if (t < 32 && !(A.lost && pass == 0)) {
            const u32 LxLy = I.LxLy;
            const int z0 = (int)div_by(c0, I.mul_p, I.sh_p), z1 = (int)div_by(c1 - 1, I.mul_p, I.sh_p);
            for (int z = z0 + t; z <= z1; z += 32) {
                const u32 lo = max(c0, (u32)z * LxLy), hi = min(c1, (u32)(z + 1) * LxLy);
                asm volatile("fence.proxy.async;" ::: "memory");   // read by copies in the next step
                __threadfence();
                atomicAdd(I.cnt + pass * I.Lz + z, hi - lo);
            }
        }
    }
    if (expired) give_up(A);
    // the last team leaves the counters as the next launch expects them
    team_barrier();
    if (t == 0) {
        __threadfence();
        const unsigned n = atomicAdd(A.work + 1, 1u);
        __threadfence();
        // 1, or 2 if the launch gave up
        t_how[team] = (n & ~kGaveUp) != (unsigned)kTeams * gridDim.x - 1u ? 0 : (n & kGaveUp ? 2 : 1);
    }
    team_barrier();
    const int how = t_how[team];
    if (how == 0) return;
    for (int k = t; k < A.n; k += kRun) {
        const PassInst &I = A.inst[k];
        const u32 base = I.cnt[3 * I.Lz] + (unsigned)A.steps * I.LxLy;
        // a launch that gave up has left slots uncounted: the counts are set to what they
        // would have reached, so that the next launch waits for its own slots alone
        for (int z = 0; how == 2 && z < 3 * I.Lz; ++z) I.cnt[z] = base;
        I.cnt[3 * I.Lz] = base;
        if (I.step_ctr) I.step_ctr[(A.parity + A.steps) & 1] = __ldcg(I.step_ctr + A.parity) + (unsigned)A.steps;
    }
    if (t == 0) {
        A.work[0] = 0u;
        A.work[1] = 0u;
    }
}

// Reciprocal of d for div_by: n / d = (t + ((n - t) >> s1)) >> s2 with
// t = floor(mul n / 2^32), exact for every 32-bit n (Granlund and Montgomery
// 1994, round-up method); s1 = 0 for d = 1 alone.
void fast_div(u32 d, u32 &mul, unsigned char &sh) {
    int l = 0;
    while ((1ull << l) < d) ++l;
    mul = (u32)((((1ull << l) - d) << 32) / d + 1);
    sh = (unsigned char)((l > 0 ? 0x80 : 0) | (l > 0 ? l - 1 : 0));
}

template <typename T, bool ADV2, bool ONE>
cudaError_t passes_k(const PassArgs *a, int grid, cudaStream_t st) {
    if (!a)   // prepare
        return cudaFuncSetAttribute(k_passes<T, ADV2, ONE>, cudaFuncAttributeMaxDynamicSharedMemorySize, pass_smem<T>());
    k_passes<T, ADV2, ONE><<<grid, kPassThreads, pass_smem<T>(), st>>>(*a);
    return cudaGetLastError();
}

template <typename T, bool ADV2>
cudaError_t passes_t(const PassArgs *a, int n, int grid, cudaStream_t st) {
    return n == 1 ? passes_k<T, ADV2, true>(a, grid, st) : passes_k<T, ADV2, false>(a, grid, st);
}

cudaError_t passes_form(const PassArgs *a, int n, int precision, int advection, int grid, cudaStream_t st) {
    switch (precision) {
        case LBFE_FP16_OFFSET: return advection ? passes_t<__half, true>(a, n, grid, st) : passes_t<__half, false>(a, n, grid, st);
        case LBFE_BF16_OFFSET:
            return advection ? passes_t<__nv_bfloat16, true>(a, n, grid, st) : passes_t<__nv_bfloat16, false>(a, n, grid, st);
        default: return advection ? passes_t<float, true>(a, n, grid, st) : passes_t<float, false>(a, n, grid, st);
    }
}

}  // namespace

// For launches of n instances (the last group of a larger batch may be one).
cudaError_t passes_prepare(int n, int precision, int advection) {
    cudaError_t e = passes_form(nullptr, n, precision, advection, 0, nullptr);
    if (e == cudaSuccess && n > 1 && n % kStepMaxInst == 1) e = passes_form(nullptr, 1, precision, advection, 0, nullptr);
    return e;
}

// Up to kPassSteps steps of every instance from state parity cur: one launch
// per 64 instances.
cudaError_t launch_passes(const LaunchCtx &c, int cur, int steps) {
    const int workers = c.num_sms * kTeams;
    for (int k0 = 0; k0 < c.n; k0 += kStepMaxInst) {
        const int k1 = k0 + kStepMaxInst < c.n ? k0 + kStepMaxInst : c.n;
        PassArgs a{};
        a.n = k1 - k0;
        a.steps = steps;
        a.parity = cur;
        a.status = c.status;
        a.work = c.status + 2;
        a.lost = c.lost_counts;
        long long cells = 0;
        for (int k = k0; k < k1; ++k) cells += c.inst_host[k].N;
        // runs of a slot: as many as leave every team a slot a pass (two slots:
        // 64^3 41.5 us against 31.8, 141 x 75 x 53 70 against 61.5; half a slot:
        // 96 x 48 x 48 34.1 against 30.2)
        int R = 1;
        while (R < kMaxRuns && cells / (kRun * 2 * R) >= workers) R *= 2;
        a.R = R;
        const long long ic = (long long)kRun * R;
        long long items = 0;
        int reach = 1;               // slots from one to the last it waits for
        for (int k = k0; k < k1; ++k) {
            const InstDev &h = c.inst_host[k];
            PassInst &d = a.inst[k - k0];
            for (int b = 0; b < 2; ++b) {
                d.f[b] = h.f[b];
                d.runs[b] = &c.maps_dev[2 * k + b].runs;
                d.C[b] = h.C[b];
                d.dens[b] = h.dens[b];
            }
            // scratch of the instance (14 S floats; the field queries use it between steps)
            d.rho = (float2 *)h.rho;
            d.pi = (float2 *)h.rho + h.S;
            d.j = h.rho + 4 * h.S;
            d.u = h.rho + 7 * h.S;
            d.cnt = h.pass_cnt;
            d.status = h.status;
            d.step_ctr = h.step_ctr;
            d.G = h.G; d.Uw = h.Uw; d.nu_A = h.nu_A; d.nu_B = h.nu_B;
            d.pi_coef = h.pi_coef; d.L2 = h.L2; d.inv_tauP = h.inv_tauP;
            d.gx = h.gx; d.gy = h.gy; d.gz = h.gz;
            d.rho0A = h.rho0[0]; d.rho0B = h.rho0[1];
            d.S = (u32)h.S;
            d.N = (u32)h.N;
            d.LxLy = (u32)(h.Lx * h.Ly);
            d.Lx = (unsigned short)h.Lx; d.Ly = (unsigned short)h.Ly; d.Lz = (unsigned short)h.Lz;
            d.visc_comp = (signed char)h.visc_comp;
            fast_div(d.LxLy, d.mul_p, d.sh_p);
            fast_div((u32)h.Lx, d.mul_x, d.sh_x);
            a.item_off[k - k0] = (int)items;
            const long long ni = (h.N + ic - 1) / ic;
            items += ni;
            // to the end of the plane after the slot's last cell's
            const long long r = (2ll * d.LxLy + ic - 1) / ic + 1;
            reach = (int)(r < ni ? (r > reach ? r : reach) : (ni > reach ? ni : reach));
        }
        a.item_off[a.n] = (int)items;
        a.items = (int)items;
        // Distance between the passes: what a slot reaches for, and half as many
        // slots as there are teams, so that most waits find their planes done
        // (no slack: 1460 us on 192 x 96 x 80; 50: 184; 100: 165; 150: 160;
        // 200: 162, the populations leave the L2 before pass X).  Small lattices
        // take what keeps a step from waiting for the one before.
        long long slack = workers / 2;
        if (slack > (items - 3ll * reach - 1) / 2) slack = (items - 3ll * reach - 1) / 2;
        if (slack < 0) slack = 0;
        a.lag_x = reach + (int)slack;
        a.lag_u = a.lag_x + reach + (int)slack;
        a.period = a.items > reach + a.lag_u + 1 ? a.items : reach + a.lag_u + 1;
        const long long slots = 3ll * ((long long)(steps - 1) * a.period + a.items + a.lag_u);
        if (slots > 0x3fffffffll) return cudaErrorInvalidValue;
        a.slots = (int)slots;
        const int grid = ((a.slots < workers ? a.slots : workers) + kTeams - 1) / kTeams;
        const cudaError_t e = passes_form(&a, a.n, c.precision, c.advection, grid, c.stream);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

int passes_steps() { return kPassSteps; }

}  // namespace lbfe
