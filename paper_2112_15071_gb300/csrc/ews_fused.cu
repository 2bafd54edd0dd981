// ews_fused.cu -- one launch per time step: the velocity pass (Eq. 1) and the
// stress pass (Eq. 2/3) of Sec. 2.3 fused, for a sponge or no absorbing
// boundary.
//
// The two-pass step moves 120 bytes per cell (velocity: 10 reads, 3 writes;
// stress: 11 reads, 6 writes) and runs at the DRAM rate on large FP32 grids.
// This step reads sigma^n, v^{n-1/2} and the medium once and writes
// v^{n+1/2} and sigma^{n+1} once: 84 bytes.  To need no exchange between CTAs
// it reads from one set of wavefields (A) and writes to a second set (B), so
// nothing a neighbour still reads is ever overwritten, and each CTA computes
// the new velocity on its 32 x TY tile plus the 2-cell ring its stress
// differences reach (36 x (TY + 4) cells, the ring computed redundantly by
// the neighbours too) and on 2 planes above and below its z-chunk.
//
// What bounds it is instruction issue and latency before DRAM, so a thread
// owns a pair of x-neighbours: shared memory is read in pairs, y- and
// z-differences and the updates are packed two-wide operations (f32x2), and
// x-differences subtract lane by lane and go on packed.  One CTA per SM, 32 x
// 24 cells: its 504 threads (16 warps) may use 128 registers, which the
// columns need, and the ring adds 31 % velocity work (32 x 8 tiles: 69 %).
// Taller tiles leave 96 or 80 registers a thread and spill (32 x 28: 35
// Gcell/s at 1024 x 1024 x 512), lower ones have fewer warps and more ring (32
// x 20 with 3 slots 60.3, 32 x 16 with 3 slots 63.9 but 58.7 at 256^3).
// Row-wise thread order keeps the
// half-warps on 16 neighbouring pairs of one row (no bank conflicts) and the
// stress threads in full warps; the ring's outer columns have threads of
// their own.  Edge masks are selects, not branches: a branch around them for
// interior tiles cut the schedule apart (55.0 against 61.3).
//
// Measured (GB300, FP32, sponge, Gcell/s, against the two passes): 1024 x
// 1024 x 512 63.4 (50.5), 256^3 61.7 (51.4), 224^3 58.4 (48.5), 192^3 60.2
// (50.0 with 32 x 4 tiles); 0.79 and 0.76 of the copy peak on 84 bytes a cell
// for the first two.  282 warp instructions per 32 cells fill 46 % of the issue
// slots; the warps wait for shared memory, copies and their own arithmetic, at
// 4 warps per scheduler.
//
// Pipeline per CTA (tile x0, y0; z-chunk z0 .. z1), step m for velocity plane
// k = z0 - 5 + m.  The copies of step m bring each field at the plane at which
// plane k completes its stencil: sxx, syy, sxy, v at k; sxz, syz, rho at k + 1;
// szz at k + 2 -- so only z-columns are held in registers, and a slot is read
// in one step only (two slots: one in use, one in flight).  The new velocity
// goes to a 5-plane shared ring, and the stress of plane k - 2 follows without
// a barrier: its x and y differences read plane k - 2, complete for two steps
// (warps count themselves past each step's velocity in an mbarrier), its
// z-columns are the thread's own; sigma^n of the cell comes from the register
// columns, lambda and mu from a three-entry TMA buffer.  The first three steps
// only fill the columns.
//
// Every mbarrier wait is bounded.  A point force (Sec. 2.4 source term of Eq.
// 1) is added to the new velocity of its tap cells before the stress uses
// them; a moment source and the receivers run after the step, on B, as in the
// two-pass loop.  The arithmetic per cell is that of the two passes, rounding
// by rounding (ews_arith.cuh).
#include <algorithm>

#include "ews_arith.cuh"
#include "ews_internal.cuh"
#include "ews_ops.cuh"
#include "ews_tma.cuh"

namespace ews {
namespace fused {
namespace {

constexpr int TX = 32;                           // tile width
constexpr int EXP = TX / 2 + 2;                  // pairs of a region row (x0-2 .. x0+33)
constexpr int VS = TX + 4;                       // row stride of the new-velocity ring
constexpr int MBW = TX + 8;                      // FP32 medium boxes: x from x0-4
constexpr int NV = 5;                            // planes of the new-velocity ring
constexpr int kMaxChunk = 1024;                  // planes of a z-chunk (its sponge gains sit in shared memory)
constexpr int NS = 2;                            // slots (one in use, the next in flight)
constexpr int NE = NS + 1;                       // entries of the medium buffer (read a phase later)

// ---- pairs of floats (x-neighbours) ----
using f2 = unsigned long long;
__device__ __forceinline__ f2 pk(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float lo(f2 a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float hi(f2 a) { return __uint_as_float((unsigned)(a >> 32)); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 dup(float a) { return pk(a, a); }
// ar::d4 on pairs
__device__ __forceinline__ f2 d4p(f2 c1, f2 c2, f2 a, f2 b, f2 c, f2 d) {
    return fma2(c1, sub2(c, b), mul2(c2, sub2(d, a)));
}
// ar::d4 along x for the pair (i, i+1) from the pairs at i-2, i, i+2: to the
// half points (DP: samples i-1 .. i+2) or to the integer points (i-2 .. i+1).
template <bool DP>
__device__ __forceinline__ f2 d4x(f2 c1, f2 c2, f2 l, f2 c, f2 r) {
    f2 in, out;
    if (DP) {
        in = pk(__fsub_rn(hi(c), lo(c)), __fsub_rn(lo(r), hi(c)));
        out = pk(__fsub_rn(lo(r), hi(l)), __fsub_rn(hi(r), lo(c)));
    } else {
        in = pk(__fsub_rn(lo(c), hi(l)), __fsub_rn(hi(c), lo(c)));
        out = pk(__fsub_rn(hi(c), lo(l)), __fsub_rn(lo(r), hi(l)));
    }
    return fma2(c1, in, mul2(c2, out));
}

__device__ __forceinline__ f2 ld2(const float* p) { return *reinterpret_cast<const f2*>(p); }
__device__ __forceinline__ void st2(float* p, f2 x) { *reinterpret_cast<f2*>(p) = x; }

// ---- shared-memory layout ----
// Slot of one step (boxes BW wide from x0 - HO): sxx, sxz rows y0-2 ..; syy
// rows y0-3 ..; syz, sxy rows y0-4 ..; szz, vx vy vz, rho rows y0-2 ...
template <int TY>
struct FL {
    static constexpr int ES = 4, HO = 4, BW = TX + 2 * HO;
    static constexpr int EY = TY + 4, NR = 16 * EY;                  // region rows; row threads
    static constexpr int NT = (EXP * EY + 31) / 32 * 32;             // threads
    static constexpr int RB = EY * BW * ES, RB3 = (EY + 3) * BW * ES, MRB = (EY + 1) * MBW * 4;
    static constexpr int SXX_ = 0, SXZ_ = r128(SXX_ + RB), SYY_ = r128(SXZ_ + RB), SYZ_ = r128(SYY_ + RB3),
                         SXY_ = r128(SYZ_ + RB3), SZZ_ = r128(SXY_ + RB3), V_ = r128(SZZ_ + RB),
                         RHO_ = r128(V_ + 3 * RB), SLOT = r128(RHO_ + MRB);
    static constexpr int FULL_TX = 3 * RB + 3 * RB3 + 3 * RB + MRB;  // all fields
    static constexpr int PRE_TX = 2 * RB + RB3 + MRB;                // sxz, syz, szz, rho
    static constexpr int LB = TX * TY * 4, MUB = (TY + 1) * MBW * 4, ENT = r128(r128(LB) + MUB);
    static constexpr int VPL = 3 * EY * VS;                          // floats of one ring plane
    static constexpr int O_V = NS * SLOT, O_E = r128(O_V + NV * VPL * 4), O_BAR = O_E + NE * ENT;
    static constexpr int O_GZ = O_BAR + r128((NS + 2) * 8), SMEM = O_GZ + (kMaxChunk + 8) * 4;
};

struct FusedMaps {
    CUtensorMap x1, y1, xy, zz, v, rho, lam, mu; // x1: sxx / sxz boxes, y1: syy / syz boxes
};

struct FusedParams {
    DevGrid g;
    DevFields fout;             // v^{n+1/2}, sigma^{n+1}
    DevMedium M;
    DevBoundary B;
    float dt, dt2, dt4;         // dt, twice it, a quarter of it
    int ntx, nty, zchunk;
    int* err;
    DevSource S;                // force taps (kind 1) of this step; else ntap 0
    const float* wavelet;
    int n;
    int sk0, sk1;               // planes of the force taps
    float* vcap;                // history slot of v^{n+1/2} (3 fields, hstride apart)
    long long hstride;
};

// First step with velocity, first that brings the medium of the stress (mu of
// plane z0), first with stress.
constexpr int M_VEL = 3, M_MED = 6, M_STR = 7;

// Issue the copies of step m (velocity plane k = z0 - 5 + m): sxz, syz, rho
// of plane k + 1 and szz of k + 2; from M_VEL on sxx, syy, sxy, v of plane k;
// from M_MED on lambda of plane k - 2 and mu of k - 1.  Medium planes clamp
// at the top.
template <int TY>
__device__ __forceinline__ void issue_step(const FusedMaps& mp, unsigned char* sm, uint64_t* bar, int x0,
                                           int y0, int z0, int m, int nz) {
    using L = FL<TY>;
    const int k = z0 - 5 + m;
    unsigned char* slot = sm + (m % NS) * L::SLOT;
    mbar_expect_tx(bar, (uint32_t)(m < M_VEL ? L::PRE_TX : m < M_MED ? L::FULL_TX : L::FULL_TX + L::LB + L::MUB));
    tma_load_4d(slot + L::SXZ_, &mp.x1, bar, x0 - L::HO, y0 - 2, k + 1, fslot(SXZ));
    tma_load_4d(slot + L::SYZ_, &mp.y1, bar, x0 - L::HO, y0 - 4, k + 1, fslot(SYZ));
    tma_load_3d(slot + L::SZZ_, &mp.zz, bar, x0 - L::HO, y0 - 2, k + 2);
    tma_load_3d(slot + L::RHO_, &mp.rho, bar, x0 - 4, y0 - 2, min(k + 1, nz - 1));
    if (m < M_VEL) return;
    tma_load_4d(slot + L::SXX_, &mp.x1, bar, x0 - L::HO, y0 - 2, k, fslot(SXX));
    tma_load_4d(slot + L::SYY_, &mp.y1, bar, x0 - L::HO, y0 - 3, k, fslot(SYY));
    tma_load_3d(slot + L::SXY_, &mp.xy, bar, x0 - L::HO, y0 - 4, k);
    tma_load_4d(slot + L::V_, &mp.v, bar, x0 - L::HO, y0 - 2, k, fslot(VX));
    if (m < M_MED) return;
    unsigned char* ent = sm + L::O_E + (m % NE) * L::ENT;
    tma_load_3d(ent, &mp.lam, bar, x0, y0, k - 2);
    tma_load_3d(ent + r128(L::LB), &mp.mu, bar, x0 - 4, y0, min(k - 1, nz - 1));
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Per-thread state across steps.
struct FQ {
    f2 zz[4], xz[4], yz[4];     // columns: szz k-1 .. k+2, sxz / syz k-2 .. k+1
    f2 xx[2], yy[2], xy[2];     // sigma^n of planes k-2, k-1 by parity (tile threads)
    f2 dz;                      // d sxz/dx + d syz/dy at plane k
    f2 bx, by, r0;              // half buoyancies and density at plane k
    f2 vzc;                     // new vz at plane k - 4 (tile threads)
    f2 mu2, mxy, ma, mb;        // 2 mu, its xy sum, mu + mu(x+1), mu + mu(y+1) at plane k - 2
    bool bad;
};

template <int BND, int TY>
struct FGeo {
    int x0, y0, z0, z1, M;
    int row, rp;                // region row, pair in the row
    int oc;                     // offset of the pair in a box that starts at row y0 - 2
    bool reg, tile;             // the thread has a region pair / a tile pair
    bool in0, in1;              // lanes inside the grid (x, y)
    bool cx0, cx1;              // lane + 1 inside the grid along x
    bool cy;                    // row + 1 inside the grid
    f2 gx;
    float gy;
    long long o;                // element of the pair in plane 0
    // values at x + 1 of the pair c with r the pair after it, clamped at the
    // grid's end
    __device__ __forceinline__ f2 next_x(f2 c, f2 r) const {
        return pk(cx0 ? hi(c) : lo(c), cx1 ? lo(r) : hi(c));
    }
    __device__ __forceinline__ FGeo(const FusedParams& P, int item) {
        using L = FL<TY>;
        const DevGrid& g = P.g;
        const int ntile = P.ntx * P.nty;
        const int tl = item % ntile;
        z0 = (item / ntile) * P.zchunk;
        z1 = min(g.nz, z0 + P.zchunk);
        M = z1 - z0 + 7;
        x0 = (tl % P.ntx) * TX;
        y0 = (tl / P.ntx) * TY;
        const int t = threadIdx.x;
        if (t < L::NR) {
            row = t >> 4;
            rp = 1 + (t & 15);
        } else {
            const int u = t - L::NR;
            row = u >> 1;
            rp = (u & 1) ? EXP - 1 : 0;
        }
        reg = t < L::EY * EXP;
        if (!reg) row = 0;
        tile = t < L::NR && row >= 2 && row < 2 + TY;
        const int i = x0 - 2 + 2 * rp, j = y0 - 2 + row;
        const bool iny = reg && j >= 0 && j < g.ny;
        in0 = iny && i >= 0 && i < g.nx;
        in1 = iny && i + 1 >= 0 && i + 1 < g.nx;
        tile = tile && in0;
        cx0 = i + 1 < g.nx;
        cx1 = i + 2 < g.nx;
        cy = j + 1 < g.ny;
        oc = row * L::BW + L::HO - 2 + 2 * rp;
        gx = dup(1.0f);
        gy = 1.0f;
        if (BND == BND_SPONGE) {
            gx = pk(in0 ? __ldg(P.B.g[0] + i) : 1.0f, in1 ? __ldg(P.B.g[0] + i + 1) : 1.0f);
            gy = iny ? __ldg(P.B.g[1] + j) : 1.0f;
        }
        o = (long long)j * g.pitch + i;
    }
};

// Slot (= its barrier) and medium entry of a step, and the phase of the
// slot's barrier.
struct Turn {
    int s = 0, ent = 0;
    uint32_t par = 0;
    __device__ __forceinline__ void next(int entry_bytes) {
        if (++s == NS) {
            s = 0;
            par ^= 1u;
        }
        ent = ent + entry_bytes == NE * entry_bytes ? 0 : ent + entry_bytes;
    }
};

// One step of the pipeline, m mod 4 == PH; STAGE 0: columns only, 1: velocity,
// 2: velocity, and the medium of plane z0, 3: velocity and stress.  ring:
// offsets of the new-velocity planes k, k-1, k-2, k-3 (floats); ent: of the
// medium entry of this step.
// CAP: v^{n+1/2} also goes to its history slot.
template <int BND, int TY, bool CAP, int PH, int STAGE>
__device__ __forceinline__ void fused_step(const FusedMaps& maps, const FusedParams& P,
                                           const FGeo<BND, TY>& G, FQ& Q, unsigned char* sm,
                                           uint64_t* bars, int m, const int (&ring)[4], const Turn& tn) {
    using L = FL<TY>;
    constexpr int BW = L::BW;
    const DevGrid& g = P.g;
    constexpr int A = (PH + 1) & 3, B = (PH + 2) & 3, C = (PH + 3) & 3, D = PH;   // oldest..newest
    constexpr int CB = NS + (PH & 1), HQ = PH & 1;                    // barrier of the warps' counts
    const int k = G.z0 - 5 + m;
    unsigned char* slot = sm + tn.s * L::SLOT;
    float* vring = reinterpret_cast<float*>(sm + L::O_V);
    const f2 c1x = dup(g.c1x), c2x = dup(g.c2x), c1y = dup(g.c1y), c2y = dup(g.c2y), c1z = dup(g.c1z), c2z = dup(g.c2z);
    const float* gz = reinterpret_cast<const float*>(sm + L::O_GZ) + m;   // gains of planes z0 - 5 + m
    // this step's copies; and every warp past its velocity phase of step m - 2
    // (so past stress m - 3): the ring plane written below is free, the one
    // read by the stress is complete
    // (after a wait that gave up the others are skipped, until the CTA leaves)
    Q.bad = Q.bad || !mbar_wait(&bars[tn.s], tn.par);
    if (STAGE > 0 || PH >= 2) Q.bad = Q.bad || !mbar_wait(&bars[CB], (uint32_t)(((m - 2) >> 1) & 1));
    // sigma^n of plane k - 2, about to leave the columns
    f2 s0, s1, s2, s3, s4, s5;
    s2 = Q.zz[D];
    s0 = Q.xx[HQ];
    s1 = Q.yy[HQ];
    s3 = Q.xy[HQ];
    {
        const float* fxz = reinterpret_cast<const float*>(slot + L::SXZ_) + G.oc;          // plane k + 1
        const float* fyz = reinterpret_cast<const float*>(slot + L::SYZ_) + G.oc + 2 * BW;
        const float* fr = reinterpret_cast<const float*>(slot + L::RHO_) + G.row * MBW + 2 + 2 * G.rp;
        const f2 cxz = ld2(fxz), cyz = ld2(fyz);
        Q.zz[D] = ld2(reinterpret_cast<const float*>(slot + L::SZZ_) + G.oc);        // plane k + 2
        Q.xz[D] = cxz;
        Q.yz[D] = cyz;
        // density and buoyancies of plane k + 1
        const f2 r1 = ld2(fr), rx = ld2(fr + 2), ry = ld2(fr + (G.cy ? MBW : 0));
        if constexpr (STAGE > 0) {
            const f2 sz = add2(Q.r0, r1);
            const float* fxx = reinterpret_cast<const float*>(slot + L::SXX_) + G.oc;
            const float* fyy = reinterpret_cast<const float*>(slot + L::SYY_) + G.oc + BW;
            const float* fxy = reinterpret_cast<const float*>(slot + L::SXY_) + G.oc + 2 * BW;
            const float* fv = reinterpret_cast<const float*>(slot + L::V_) + G.oc;
            const f2 cxx = ld2(fxx), cyy = ld2(fyy), cxy = ld2(fxy);
            Q.xx[HQ] = cxx;
            Q.yy[HQ] = cyy;
            Q.xy[HQ] = cxy;
            f2 dxx = d4x<true>(c1x, c2x, ld2(fxx - 2), cxx, ld2(fxx + 2));
            f2 dxy = d4p(c1y, c2y, ld2(fxy - 2 * BW), ld2(fxy - BW), cxy, ld2(fxy + BW));
            f2 dxz = d4p(c1z, c2z, Q.xz[A], Q.xz[B], Q.xz[C], Q.xz[D]);
            f2 dyx = d4x<false>(c1x, c2x, ld2(fxy - 2), cxy, ld2(fxy + 2));
            f2 dyy = d4p(c1y, c2y, ld2(fyy - BW), cyy, ld2(fyy + BW), ld2(fyy + 2 * BW));
            f2 dyz = d4p(c1z, c2z, Q.yz[A], Q.yz[B], Q.yz[C], Q.yz[D]);
            f2 dzz = d4p(c1z, c2z, Q.zz[A], Q.zz[B], Q.zz[C], Q.zz[D]);
            // (2 dt) r with r = 1 / (r0 + r1) has the bits of dt (2 r)
            const f2 bz = pk(ar::rcp(lo(sz)), ar::rcp(hi(sz)));
            f2 vx = fma2(mul2(dup(P.dt2), Q.bx), add2(add2(dxx, dxy), dxz), ld2(fv));
            f2 vy = fma2(mul2(dup(P.dt2), Q.by), add2(add2(dyx, dyy), dyz), ld2(fv + L::RB / L::ES));
            f2 vz = fma2(mul2(dup(P.dt2), bz), add2(Q.dz, dzz), ld2(fv + 2 * (L::RB / L::ES)));
            if (BND == BND_SPONGE) {
                const f2 gs = mul2(mul2(G.gx, dup(gz[0])), dup(G.gy));
                vx = mul2(vx, gs); vy = mul2(vy, gs); vz = mul2(vz, gs);
            }
            const bool kin = k >= 0 && k < g.nz;         // zero outside the grid
            const bool i0 = kin && G.in0, i1 = kin && G.in1;
            vx = pk(i0 ? lo(vx) : 0.0f, i1 ? hi(vx) : 0.0f);
            vy = pk(i0 ? lo(vy) : 0.0f, i1 ? hi(vy) : 0.0f);
            vz = pk(i0 ? lo(vz) : 0.0f, i1 ? hi(vz) : 0.0f);
            if (G.tile && k >= G.z0 && k < G.z1) {
                const long long o = (long long)k * g.plane + G.o;
                st2(P.fout.f[VX] + o, vx);
                st2(P.fout.f[VY] + o, vy);
                st2(P.fout.f[VZ] + o, vz);
                if constexpr (CAP) {
                    st2(P.vcap + o, vx);
                    st2(P.vcap + P.hstride + o, vy);
                    st2(P.vcap + 2 * P.hstride + o, vz);
                }
            }
            if (G.reg) {
                float* vn = vring + ring[0] + G.row * VS + 2 * G.rp;
                *reinterpret_cast<f2*>(vn) = vx;
                *reinterpret_cast<f2*>(vn + L::EY * VS) = vy;
                *reinterpret_cast<f2*>(vn + 2 * L::EY * VS) = vz;
            }
        }
        Q.r0 = r1;
        const f2 sx = add2(r1, G.next_x(r1, rx)), sy = add2(r1, ry);
        Q.bx = pk(ar::rcp(lo(sx)), ar::rcp(hi(sx)));
        Q.by = pk(ar::rcp(lo(sy)), ar::rcp(hi(sy)));
        f2 dzx = d4x<false>(c1x, c2x, ld2(fxz - 2), cxz, ld2(fxz + 2));
        f2 dzy = d4p(c1y, c2y, ld2(fyz - 2 * BW), ld2(fyz - BW), cyz, ld2(fyz + BW));
        Q.dz = add2(dzx, dzy);
    }
    s4 = Q.xz[A];                                    // sxz, syz of plane k - 2
    s5 = Q.yz[A];
    // the warp is done with this step's slot and its part of the ring plane
    __syncwarp();
    if ((threadIdx.x & 31) == 0) mbar_arrive(&bars[CB]);
    // the last warp, which has no stress to compute, refills the slot for step
    // m + NS once every warp is
    if (threadIdx.x == L::NT - 32 && m + NS < G.M) {
        Q.bad = Q.bad || !mbar_wait(&bars[CB], (uint32_t)((m >> 1) & 1));
        issue_step<TY>(maps, sm, &bars[tn.s], G.x0, G.y0, G.z0, m + NS, g.nz);
    }
    // point force of step n on its tap cells inside the region
    if (STAGE > 0 && k >= P.sk0 && k <= P.sk1) {     // uniform across the CTA
        __syncthreads();
        if ((int)threadIdx.x < P.S.ntap) {
            const Tap tp = P.S.tap[threadIdx.x];
            const int ex = tp.i - (G.x0 - 2), ey = tp.j - (G.y0 - 2);
            if (tp.k == k && ex >= 0 && ex < TX + 4 && ey >= 0 && ey < L::EY) {
                float amp = __fmul_rn(tp.w, __ldg(P.wavelet + P.n));
                amp *= ops::buoy(P.M, g, tp.q - VX, tp.i, tp.j, tp.k);
                amp *= ops::gain(P.B, tp.i, tp.j, tp.k);
                float* v = vring + ring[0] + (tp.q - VX) * L::EY * VS + ey * VS + ex;
                const float x = __fadd_rn(*v, amp);
                *v = x;
                if (k >= G.z0 && k < G.z1 && ex >= 2 && ex < 2 + TX && ey >= 2 && ey < 2 + TY) {
                    float* f = tp.q == VX ? P.fout.f[VX] : tp.q == VY ? P.fout.f[VY] : P.fout.f[VZ];
                    f[ops::cidx(g, tp.i, tp.j, tp.k)] = x;
                    if constexpr (CAP) P.vcap[(tp.q - VX) * P.hstride + ops::cidx(g, tp.i, tp.j, tp.k)] = x;
                }
            }
        }
        __syncthreads();
    }
    // ---- stress of plane k - 2 at the tile pair (Eq. 2/3) ----
    if constexpr (STAGE >= 2) {
        if (G.tile) {
            const unsigned char* ent = sm + L::O_E + tn.ent;
            const float* hm = reinterpret_cast<const float*>(ent + r128(L::LB)) + (G.row - 2) * MBW + 2 + 2 * G.rp;
            const float* hy = hm + (G.cy ? MBW : 0);
            // mu of plane k - 1 and its x, y and xy neighbours
            const f2 m1 = ld2(hm), m1r = ld2(hm + 2), my = ld2(hy), myr = ld2(hy + 2);
            const f2 mx = G.next_x(m1, m1r), mxy4 = G.next_x(my, myr);
            const f2 na = add2(m1, mx), nb = add2(m1, my);
            const int e = G.row * VS + 2 * G.rp;
            const float* v2 = vring + ring[2] + e;                                   // plane k - 2
            const float* v3 = vring + ring[3] + e;
            const float* v1 = vring + ring[1] + e;
            const float* v0 = vring + ring[0] + e;
            constexpr int FS = L::EY * VS;
            const f2 vz3 = ld2(v3 + 2 * FS), czv = ld2(v2 + 2 * FS);
            if constexpr (STAGE == 3) {
                const f2 cvx = ld2(v2), cvy = ld2(v2 + FS);
                f2 exx = d4x<false>(c1x, c2x, ld2(v2 - 2), cvx, ld2(v2 + 2));
                f2 vxy = d4p(c1y, c2y, ld2(v2 - VS), cvx, ld2(v2 + VS), ld2(v2 + 2 * VS));
                f2 vxz = d4p(c1z, c2z, ld2(v3), cvx, ld2(v1), ld2(v0));
                f2 eyy = d4p(c1y, c2y, ld2(v2 + FS - 2 * VS), ld2(v2 + FS - VS), cvy, ld2(v2 + FS + VS));
                f2 vyx = d4x<true>(c1x, c2x, ld2(v2 + FS - 2), cvy, ld2(v2 + FS + 2));
                f2 vyz = d4p(c1z, c2z, ld2(v3 + FS), cvy, ld2(v1 + FS), ld2(v0 + FS));
                f2 ezz = d4p(c1z, c2z, Q.vzc, vz3, czv, ld2(v1 + 2 * FS));
                f2 vzx = d4x<true>(c1x, c2x, ld2(v2 + 2 * FS - 2), czv, ld2(v2 + 2 * FS + 2));
                f2 vzy = d4p(c1y, c2y, ld2(v2 + 2 * FS - VS), czv, ld2(v2 + 2 * FS + VS), ld2(v2 + 2 * FS + 2 * VS));
                const f2 lam = ld2(reinterpret_cast<const float*>(ent) + (G.row - 2) * TX + 2 * (G.rp - 1));
                const f2 l2m = add2(Q.mu2, lam);
                // sums of four: (dt / 4) times the sum has the bits of dt times the mean
                const f2 mxz = add2(add2(Q.ma, m1), mx), myz = add2(add2(Q.mb, m1), my);
                s0 = fma2(dup(P.dt), fma2(l2m, exx, mul2(lam, add2(eyy, ezz))), s0);
                s1 = fma2(dup(P.dt), fma2(l2m, eyy, mul2(lam, add2(exx, ezz))), s1);
                s2 = fma2(dup(P.dt), fma2(l2m, ezz, mul2(lam, add2(exx, eyy))), s2);
                s3 = fma2(mul2(dup(P.dt4), Q.mxy), add2(vxy, vyx), s3);
                s4 = fma2(mul2(dup(P.dt4), mxz), add2(vxz, vzx), s4);
                s5 = fma2(mul2(dup(P.dt4), myz), add2(vyz, vzy), s5);
                if (BND == BND_SPONGE) {
                    const f2 gs = mul2(mul2(G.gx, dup(gz[-2])), dup(G.gy));
                    s0 = mul2(s0, gs); s1 = mul2(s1, gs); s2 = mul2(s2, gs);
                    s3 = mul2(s3, gs); s4 = mul2(s4, gs); s5 = mul2(s5, gs);
                }
                if (!G.in1) {              // the padding stays zero
                    s0 = pk(lo(s0), 0.f); s1 = pk(lo(s1), 0.f); s2 = pk(lo(s2), 0.f);
                    s3 = pk(lo(s3), 0.f); s4 = pk(lo(s4), 0.f); s5 = pk(lo(s5), 0.f);
                }
                const long long o = (long long)(k - 2) * g.plane + G.o;
                st2(P.fout.f[SXX] + o, s0);
                st2(P.fout.f[SYY] + o, s1);
                st2(P.fout.f[SZZ] + o, s2);
                st2(P.fout.f[SXY] + o, s3);
                st2(P.fout.f[SXZ] + o, s4);
                st2(P.fout.f[SYZ] + o, s5);
            }
            Q.vzc = vz3;
            Q.mu2 = add2(m1, m1);
            Q.ma = na;
            Q.mb = nb;
            Q.mxy = add2(add2(na, my), mxy4);
        }
    }
}

template <int BND, int TY, bool CAP>
__global__ void __launch_bounds__(FL<TY>::NT, 1) k_fused(const __grid_constant__ FusedMaps maps,
                                                           const __grid_constant__ FusedParams P) {
    using L = FL<TY>;
    extern __shared__ __align__(128) unsigned char sm[];
    // bars[0..NS-1]: copies of a step arrived; the last two: warps past its velocity phase
    uint64_t* bars = reinterpret_cast<uint64_t*>(sm + L::O_BAR);
    const FGeo<BND, TY> G(P, (int)blockIdx.x);
    if (threadIdx.x == L::NT - 32) {
        for (int s = 0; s < NS + 2; ++s) mbar_init(&bars[s], s < NS ? 1 : L::NT / 32);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        for (int s = 0; s < NS; ++s) issue_step<TY>(maps, sm, &bars[s], G.x0, G.y0, G.z0, s, P.g.nz);
    }
    if (BND == BND_SPONGE)
        for (int q = threadIdx.x; q < G.M; q += L::NT)
            reinterpret_cast<float*>(sm + L::O_GZ)[q] = __ldg(P.B.g[2] + min(max(G.z0 - 5 + q, 0), P.g.nz - 1));
    __syncthreads();
    FQ Q;
#pragma unroll
    for (int q = 0; q < 4; ++q) Q.zz[q] = Q.xz[q] = Q.yz[q] = 0;
    Q.xx[0] = Q.xx[1] = Q.yy[0] = Q.yy[1] = Q.xy[0] = Q.xy[1] = 0;
    Q.dz = Q.bx = Q.by = Q.r0 = Q.vzc = Q.mu2 = Q.mxy = Q.ma = Q.mb = 0;
    Q.bad = false;
    int ring[4] = {0, 4 * L::VPL, 3 * L::VPL, 2 * L::VPL};            // planes k .. k - 3
    Turn tn;
    auto next = [&]() {
        const int nw = ring[0] + L::VPL == NV * L::VPL ? 0 : ring[0] + L::VPL;
        ring[3] = ring[2];
        ring[2] = ring[1];
        ring[1] = ring[0];
        ring[0] = nw;
        tn.next(L::ENT);
    };
    fused_step<BND, TY, CAP, 0, 0>(maps, P, G, Q, sm, bars, 0, ring, tn); next();
    fused_step<BND, TY, CAP, 1, 0>(maps, P, G, Q, sm, bars, 1, ring, tn); next();
    fused_step<BND, TY, CAP, 2, 0>(maps, P, G, Q, sm, bars, 2, ring, tn); next();
    fused_step<BND, TY, CAP, 3, 1>(maps, P, G, Q, sm, bars, 3, ring, tn); next();
    fused_step<BND, TY, CAP, 0, 1>(maps, P, G, Q, sm, bars, 4, ring, tn); next();
    fused_step<BND, TY, CAP, 1, 1>(maps, P, G, Q, sm, bars, 5, ring, tn); next();
    fused_step<BND, TY, CAP, 2, 2>(maps, P, G, Q, sm, bars, 6, ring, tn); next();
    fused_step<BND, TY, CAP, 3, 3>(maps, P, G, Q, sm, bars, 7, ring, tn); next();
    int m = M_STR + 1;
    bool stop = __syncthreads_or(Q.bad);
    while (m < G.M && !stop) {
        fused_step<BND, TY, CAP, 0, 3>(maps, P, G, Q, sm, bars, m, ring, tn);
        next();
        if (++m < G.M) {
            fused_step<BND, TY, CAP, 1, 3>(maps, P, G, Q, sm, bars, m, ring, tn);
            next();
            if (++m < G.M) {
                fused_step<BND, TY, CAP, 2, 3>(maps, P, G, Q, sm, bars, m, ring, tn);
                next();
                if (++m < G.M) {
                    fused_step<BND, TY, CAP, 3, 3>(maps, P, G, Q, sm, bars, m, ring, tn);
                    next();
                    ++m;
                }
            }
        }
        // a wait that gave up ends the CTA here; one barrier in 64 steps
        if ((m & 63) < 4 || m >= G.M) stop = __syncthreads_or(Q.bad);
    }
    if (stop && threadIdx.x == 0) {          // record, and let the copies in flight land (bounded)
        atomicOr(P.err, 1);
        for (int q = m; q < m + NS && q < G.M; ++q)
            if (!mbar_wait(&bars[q % NS], (uint32_t)((q / NS) & 1))) break;
    }
}

template <int TY>
bool encode_fused(FusedMaps* fm, const DevGrid& g, const DevFields& F, const DevMedium& M) {
    using L = FL<TY>;
    const CUtensorMapDataType f32 = CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    const char* f0 = (const char*)F.f[SXX];                                    // slot 0
    const long long fsb = (const char*)F.f[SXZ] - (const char*)F.f[SXX];
    for (int q = 0; q < NFIELD; ++q)
        if ((const char*)F.f[q] - f0 != fslot(q) * fsb) return false;
    bool ok = true;
    ok &= encode4(&fm->x1, g, f0, f32, L::ES, fsb, NFIELD, L::BW, L::EY, 1);
    ok &= encode4(&fm->y1, g, f0, f32, L::ES, fsb, NFIELD, L::BW, L::EY + 3, 1);
    ok &= encode(&fm->xy, g, F.f[SXY], f32, L::ES, L::BW, L::EY + 3);
    ok &= encode(&fm->zz, g, F.f[SZZ], f32, L::ES, L::BW, L::EY);
    ok &= encode4(&fm->v, g, f0, f32, L::ES, fsb, NFIELD, L::BW, L::EY, 3);
    ok &= encode(&fm->rho, g, M.rho, f32, 4, MBW, L::EY + 1);
    ok &= encode(&fm->lam, g, M.lam, f32, 4, TX, TY);
    ok &= encode(&fm->mu, g, M.mu, f32, 4, MBW, TY + 1);
    return ok;
}

}  // namespace

struct FusedPlan {
    FusedMaps dir[2];             // reading A (dir 0) or B (dir 1)
    DevFields f[2];
    int kind = 0;
    int ty = 0, nt = 0, smem = 0;
    void (*kern)(FusedMaps, FusedParams) = nullptr;
    void (*kern_cap)(FusedMaps, FusedParams) = nullptr;   // also capturing the history
    int ntx = 0, nty = 0, zchunk = 0, grid = 0;
};

namespace {
template <int TY>
cudaError_t plan_for(FusedPlan* p, const DevGrid& g, const DevFields& A, const DevFields& Bf, const DevMedium& M,
                     const DevBoundary& B) {
    using L = FL<TY>;
    static_assert(L::SMEM <= 227 * 1024, "one CTA's shared memory");
    p->kern = B.kind == BND_SPONGE ? k_fused<BND_SPONGE, TY, false> : k_fused<BND_NONE, TY, false>;
    p->kern_cap = B.kind == BND_SPONGE ? k_fused<BND_SPONGE, TY, true> : k_fused<BND_NONE, TY, true>;
    p->ty = TY;
    p->nt = L::NT;
    p->smem = L::SMEM;
    if (!encode_fused<TY>(&p->dir[0], g, A, M) || !encode_fused<TY>(&p->dir[1], g, Bf, M))
        return cudaErrorInvalidValue;
    return cudaSuccess;
}
}  // namespace

bool fused_supported(const DevGrid& g, const DevBoundary& B, int storage) {
    return storage == EWS_STORAGE_F32 && (B.kind == BND_SPONGE || B.kind == BND_NONE) &&
           g.fs == kNoSurface && !g.cm[0];
}

cudaError_t fused_plan_create(const DevGrid& g, const DevFields& A, const DevFields& Bf,
                              const DevMedium& M, const DevBoundary& B, FusedPlan** out) {
    FusedPlan* p = new FusedPlan();
    p->kind = B.kind;
    p->f[0] = A;
    p->f[1] = Bf;
    int dev = 0, sms = 0, occ = 0;
    cudaError_t e = plan_for<24>(p, g, A, Bf, M, B);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(p->kern, cudaFuncAttributeMaxDynamicSharedMemorySize, p->smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(p->kern_cap, cudaFuncAttributeMaxDynamicSharedMemorySize, p->smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, p->kern, p->nt, p->smem);
    if (e == cudaSuccess && occ < 1) e = cudaErrorInvalidConfiguration;
    if (e != cudaSuccess) {
        delete p;
        return e;
    }
    p->ntx = (g.nx + TX - 1) / TX;
    p->nty = (g.ny + p->ty - 1) / p->ty;
    const long long ntile = (long long)p->ntx * p->nty;
    // a chunk runs 4 more velocity planes than it has planes and 3 light steps
    p->zchunk = std::min(kMaxChunk, chunk_planes(ntile, (long long)sms * occ, g.nz, 8, 6));
    p->grid = (int)(ntile * ((g.nz + p->zchunk - 1) / p->zchunk));
    *out = p;
    return cudaSuccess;
}

void fused_plan_destroy(FusedPlan* p) { delete p; }

cudaError_t launch_fused(const FusedPlan* p, int dir, const DevGrid& g, const DevMedium& M,
                         const DevBoundary& B, float dt, const DevSource& S, const float* wavelet, int n,
                         float* vcap, long long hstride, int* err, cudaStream_t st) {
    FusedParams P{};
    P.g = g;
    P.fout = p->f[dir ^ 1];
    P.M = M;
    P.B = B;
    P.dt = dt;
    P.dt2 = 2.0f * dt;
    P.dt4 = 0.25f * dt;
    P.ntx = p->ntx;
    P.nty = p->nty;
    P.zchunk = p->zchunk;
    P.err = err;
    P.S.kind = -1;
    P.S.ntap = 0;
    P.sk0 = 1 << 30;
    P.sk1 = -(1 << 30);
    if (S.kind == 1 && S.ntap > 0) {
        P.S = S;
        P.wavelet = wavelet;
        P.n = n;
        for (int t = 0; t < S.ntap; ++t) {
            P.sk0 = std::min(P.sk0, S.tap[t].k);
            P.sk1 = std::max(P.sk1, S.tap[t].k);
        }
    }
    P.vcap = vcap;
    P.hstride = hstride;
    (vcap ? p->kern_cap : p->kern)<<<p->grid, p->nt, p->smem, st>>>(p->dir[dir], P);
    return cudaGetLastError();
}

}  // namespace fused
}  // namespace ews
