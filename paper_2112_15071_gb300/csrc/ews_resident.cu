// ews_resident.cu -- the whole time loop of a small grid in one cooperative
// launch, with the wavefields resident on the SMs.
//
// On a grid of up to about 70^3 cells a time step of the two passes takes
// microseconds, most of them launch gaps, pipeline fill and the tail of each
// kernel.  Here each CTA (one per SM) owns one block of at most 16 x 16 x 12
// cells for all steps of the call.  Its 9 fields, with a 2-cell halo, stay in
// shared memory and the 8 medium values of each cell in registers.  A step is two phases, velocity (Eq. 1) and
// stress (Eq. 2/3).  In each a CTA receives the halo layers its differences
// reach from its face neighbours (the stencil is a star, so only faces),
// updates its cells and sends its new face layers to them.
//
// Exchange: every halo value travels as one 64-bit word, the value and a tag
// that counts the steps, stored by the sender straight into the receiver's
// inbox and polled there, so a phase costs one store-to-load latency; with
// plain halo loads behind a released counter (fence, counter, load: three
// round trips) a step of 64^3 took 10.3 us.  One inbox per exchange is
// enough: a sender writes sigma of step n only after it has received the
// neighbour's velocity of step n, which the neighbour sends after it has
// read sigma of step n - 1; the same holds for the velocity.  Tags never
// repeat (the caller advances `epoch` by the steps of each launch).
//
// All CTAs are resident at once (cooperative launch), so every awaited value
// is sent by a running CTA; each wait is bounded all the same and ends in the
// error flag.  The global fields are read at the start and written at the
// end of the launch.  Receivers: the owner of each tap cell writes v^{n+1/2}
// of its taps to a staging row per step, and k_resident_record sums the 8
// taps of every sample afterwards in the order of the receiver kernel.  The
// arithmetic is that of the passes (ews_arith.cuh), rounding by rounding.
#include <algorithm>
#include <new>
#include <vector>

#include "ews_arith.cuh"
#include "ews_internal.cuh"
#include "ews_ops.cuh"

namespace ews {
namespace {

constexpr int MX = 16, MY = 16;                  // largest block in x and y
constexpr int SX = MX + 4, SP = SX * (MY + 4);   // shared-memory strides (row, plane)
constexpr int MAXZ = 12;                         // largest block in z
// Elements of one field in shared memory, by the planes of a block (the
// 1024-thread kernels serve blocks of at most 4, the 512-thread ones of 5 to 8
// and the 768-thread ones of 9 to 12 planes).
constexpr int fcap(int lz) { return SP * (lz <= 4 ? 8 : lz <= 8 ? 12 : MAXZ + 4); }
constexpr int COLS = MX * MY;                    // threads of one z-group
static_assert(NFIELD * fcap(MAXZ) * 4 + 1024 <= 227 * 1024 && (NFIELD * fcap(4) + 18 * 1024) * 4 + 1024 <= 227 * 1024 && (NFIELD + 3) * fcap(8) * 4 + 1024 <= 227 * 1024,
              "fields (and the history's, reverse) fit one CTA's shared memory");

struct ResParams {
    DevGrid g;
    DevFields F;
    DevMedium M;
    DevBoundary B;
    float dt;
    DevSource S;
    const float* wavelet;
    int n0, nsteps;
    unsigned long long* inbox;                   // [CTAs][2 exchanges][9][lines]
    unsigned epoch;                              // tag of the step before n0
    int* err;
    int nbx, nby, nbz, lcap0, lcap1, lines;      // blocks; lines of x, of x and y, of all faces
    const int2* tlist;                           // receiver taps by CTA: (shared offset, tap)
    const int* tstart;                           // [CTAs + 1] ranges of tlist
    float* stage;                                // [nsteps][ntap] v at the taps, or null
    int ntap;
    float* vcap;                                 // history slot of step n0 (3 fields), or null
    // reverse sweep (n0 + nsteps - 1 down to n0): the history, slot n - h0 + 1
    // holding v^{n+1/2}; whether slot n0 + nsteps - h0 + 1 exists; the
    // accumulators, added to FP64 every `flush` steps; the residual
    const float* vhist;
    int h0, vnext, flush;
    AdjFields A;
    float gdt;
    const float* sadj;
    int ld;
    const Tap* taps;
    float* coef;                                 // [ntap] scratch, by place in tlist
    long long fstride;                           // elements between fields
    unsigned long long wait_ns;
    int mute;                                    // CTA that leaves at once (testing), or -1
};

__device__ __forceinline__ unsigned long long inbox_load(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void inbox_store(unsigned long long* p, float x, unsigned tag) {
    const unsigned long long v = ((unsigned long long)tag << 32) | __float_as_uint(x);
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ unsigned long long clock_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// First cell and length of block b of nb along an axis of n cells.
__host__ __device__ __forceinline__ int block_lo(int n, int nb, int b) {
    return (int)((long long)n * b / nb);
}

// One halo line of a CTA's face: the layers -2, -1, L, L + 1 along `axis`
// beside one cell of the face.  Neighbours along the axis have the same
// line at the same place of their inbox.
struct HaloLine {
    int so, ss, len;     // shared offset of the cell at 0 along the axis, stride, block length
    int axis;            // -1: the thread has no line
    int go, gs;          // the same in the global fields (first step only)
    int in;              // the line's place in this CTA's inbox (first exchange, value 0)
    int lo, hi;          // and in the inbox of the neighbour below / above; -1: none
};
// The three fields whose differences run along the line's axis: the first
// goes to the half points in the velocity phase (layers -1, L, L + 1) and to
// the integer points in the stress phase (-2, -1, L), the others the other
// way round.
template <bool VEL>
__device__ __forceinline__ void line_fields(int axis, int q[3]) {
    if (VEL) {
        q[0] = axis == 0 ? SXX : axis == 1 ? SYY : SZZ;
        q[1] = axis == 2 ? SXZ : SXY;
        q[2] = axis == 0 ? SXZ : SYZ;
    } else {
        q[0] = axis;
        q[1] = axis == 0 ? VY : VX;
        q[2] = axis == 2 ? VY : VZ;
    }
}
// Place in the shared field of value v (0..2) of a line: 0 is layer -1, 2 is
// layer L, 1 is layer L + 1 (to half points) or -2.
template <bool DP>
__device__ __forceinline__ int layer_at(const HaloLine& h, int v) {
    return v == 0 ? -1 : v == 2 ? h.len : DP ? h.len + 1 : -2;
}
template <bool DP>
__device__ __forceinline__ bool from_hi(int v) { return v == 2 || (DP && v == 1); }

// Halo layers of the first step, from the global fields.
template <bool VEL, int FCAP>
__device__ __forceinline__ void halo_first(const HaloLine& h, const ResParams& P, float* sm) {
    if (h.axis < 0) return;
    int q[3];
    line_fields<VEL>(h.axis, q);
#pragma unroll
    for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const bool hi = (f == 0) == VEL ? from_hi<true>(v) : from_hi<false>(v);
            const int at = (f == 0) == VEL ? layer_at<true>(h, v) : layer_at<false>(h, v);
            if ((hi ? h.hi : h.lo) >= 0) sm[q[f] * FCAP + h.so + at * h.ss] = __ldcg(P.F.f[q[f]] + h.go + at * h.gs);
        }
}
// Receive the layers of one exchange (VEL: sigma, for the velocity phase).
template <bool VEL, int FCAP>
__device__ __forceinline__ bool halo_recv(const HaloLine& h, const ResParams& P, float* sm, unsigned tag) {
    if (h.axis < 0) return true;
    const unsigned long long* in = P.inbox + h.in + (VEL ? 0 : 9 * P.lines);
    unsigned need = 0;
#pragma unroll
    for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const bool hi = (f == 0) == VEL ? from_hi<true>(v) : from_hi<false>(v);
            if ((hi ? h.hi : h.lo) >= 0) need |= 1u << (3 * f + v);
        }
    unsigned long long x[9] = {};
    unsigned long long t0 = 0;
    for (unsigned it = 0;; ++it) {
#pragma unroll
        for (int e = 0; e < 9; ++e)
            if ((need >> e) & 1u) x[e] = inbox_load(in + e * P.lines);
        bool all = true;
#pragma unroll
        for (int e = 0; e < 9; ++e)
            if (((need >> e) & 1u) && (unsigned)(x[e] >> 32) != tag) all = false;
        if (all) break;
        if ((it & 255u) == 255u) {                                   // off the usual path: a round trip of its own
            if (*(volatile int*)P.err & 3) return false;             // another CTA gave up
            const unsigned long long now = clock_ns();
            if (it == 255u) t0 = now;
            if (now - t0 > P.wait_ns) {
                atomicOr(P.err, 1);
                return false;
            }
        }
    }
    int q[3];
    line_fields<VEL>(h.axis, q);
#pragma unroll
    for (int f = 0; f < 3; ++f)
#pragma unroll
        for (int v = 0; v < 3; ++v)
            if ((need >> (3 * f + v)) & 1u) {
                const int at = (f == 0) == VEL ? layer_at<true>(h, v) : layer_at<false>(h, v);
                sm[q[f] * FCAP + h.so + at * h.ss] = __uint_as_float((unsigned)x[3 * f + v]);
            }
    return true;
}
// Send this CTA's face layers of one exchange: to the neighbour below, whose
// layers L and L + 1 are this CTA's cells 0 and 1, and to the one above,
// whose layers -1 and -2 are the last two.
template <bool VEL, int FCAP>
__device__ __forceinline__ void halo_send(const HaloLine& h, const ResParams& P, const float* sm, unsigned tag) {
    if (h.axis < 0) return;
    int q[3];
    line_fields<VEL>(h.axis, q);
#pragma unroll
    for (int f = 0; f < 3; ++f) {
        const float* s = sm + q[f] * FCAP + h.so;
#pragma unroll
        for (int v = 0; v < 3; ++v) {
            const bool hi = (f == 0) == VEL ? from_hi<true>(v) : from_hi<false>(v);   // as the receiver sees it
            const int to = hi ? h.lo : h.hi;
            const int at = hi ? (v == 2 ? 0 : 1) : h.len - (v == 0 ? 1 : 2);
            if (to >= 0)
                inbox_store(P.inbox + to + ((VEL ? 0 : 9) + 3 * f + v) * P.lines, s[at * h.ss], tag);
        }
    }
}

// ADJ: the reverse sweep in transformed variables (F are the adjoint fields,
// dt is negative): the velocity phase also accumulates the gradient products
// of the pass k_velocity<M_GRAD>, with the forward velocity's history staged
// as three more shared fields, and the residual is injected after it.
template <int BND, int FS, int CPT, int MAXT, bool ADJ = false>
__global__ void __launch_bounds__(MAXT, 1) k_resident(const __grid_constant__ ResParams P) {
    constexpr int FCAP = fcap(MAXT == 768 ? MAXZ : MAXT == 512 ? 8 : 4);
    // With a cell per thread the C-PML memory variables of the block fit shared
    // memory too (18 rows of MAXT); larger blocks keep them in global memory.
    constexpr bool PSM = BND == BND_CPML && CPT == 1;
    constexpr int H0 = NFIELD;                   // first history field
    extern __shared__ __align__(16) float sm[];
    __shared__ float s_amp[kMaxSrcTaps][2];      // buoyancy, gain of the block's source taps
    __shared__ int s_off[kMaxSrcTaps];           // their shared offset, -1: not in this block
    __shared__ int s_src;
    const DevGrid& g = P.g;
    const int t = threadIdx.x, NT = blockDim.x, cta = blockIdx.x;
    if (cta == P.mute) return;
    const int bi = cta % P.nbx, bj = (cta / P.nbx) % P.nby, bk = cta / (P.nbx * P.nby);
    const int i0 = block_lo(g.nx, P.nbx, bi), j0 = block_lo(g.ny, P.nby, bj), k0 = block_lo(g.nz, P.nbz, bk);
    const int LX = block_lo(g.nx, P.nbx, bi + 1) - i0, LY = block_lo(g.ny, P.nby, bj + 1) - j0,
              LZ = block_lo(g.nz, P.nbz, bk + 1) - k0;
    // column of the thread: half-warps take rows j and j + 4, whose offsets
    // (4 x 20 words) fall on the other 16 banks
    const int lane = t & 31, w = (t >> 5) & 7;
    const int ci = lane & 15, cj = (w & 3) + 8 * (w >> 2) + 4 * (lane >> 4);
    const int kz = (t / COLS) * CPT;             // first of the thread's CPT cells along z
    const bool col = ci < LX && cj < LY;
    const int nc = col ? min(CPT, LZ - kz) : 0;  // cells of the thread (may be <= 0)
    const int so = (kz + 2) * SP + (cj + 2) * SX + ci + 2;
    const int gi = i0 + ci, gj = j0 + cj, gk = k0 + kz;
    const int plane = (int)g.plane;
    const int go = gk * plane + gj * g.pitch + gi;

    for (int x = t; x < (NFIELD + (ADJ ? 3 : 0)) * FCAP; x += NT) sm[x] = 0.0f;
    if (t == 0) s_src = 0;
    __syncthreads();
    // medium of the thread's cells at their staggered points; sponge gains
    float mb[CPT][3], ml[CPT], mm[CPT], ms[CPT][3], mg[CPT];
#pragma unroll
    for (int c = 0; c < CPT; ++c) {
        if (c >= nc) continue;
        const int k = gk + c;
        if (g.cm[0]) {
            const float fi = (float)gi, fj = (float)gj, fk = (float)k;
            mb[c][0] = __fdividef(1.0f, coarse_at(g, 2, fi + 0.5f, fj, fk));
            mb[c][1] = __fdividef(1.0f, coarse_at(g, 2, fi, fj + 0.5f, fk));
            mb[c][2] = __fdividef(1.0f, coarse_at(g, 2, fi, fj, fk + 0.5f));
            ml[c] = coarse_at(g, 0, fi, fj, fk);
            mm[c] = coarse_at(g, 1, fi, fj, fk);
            ms[c][0] = coarse_at(g, 1, fi + 0.5f, fj + 0.5f, fk);
            ms[c][1] = coarse_at(g, 1, fi + 0.5f, fj, fk + 0.5f);
            ms[c][2] = coarse_at(g, 1, fi, fj + 0.5f, fk + 0.5f);
        } else {
            const float r0 = ops::med(P.M.rho, g, gi, gj, k);
            mb[c][0] = ar::buoyancy(r0, ops::med(P.M.rho, g, gi + 1, gj, k));
            mb[c][1] = ar::buoyancy(r0, ops::med(P.M.rho, g, gi, gj + 1, k));
            mb[c][2] = ar::buoyancy(r0, ops::med(P.M.rho, g, gi, gj, k + 1));
            ml[c] = ops::med(P.M.lam, g, gi, gj, k);
            const float m0 = ops::med(P.M.mu, g, gi, gj, k), mx = ops::med(P.M.mu, g, gi + 1, gj, k),
                        my = ops::med(P.M.mu, g, gi, gj + 1, k), mz = ops::med(P.M.mu, g, gi, gj, k + 1);
            const float mxy = ops::med(P.M.mu, g, gi + 1, gj + 1, k), mxz = ops::med(P.M.mu, g, gi + 1, gj, k + 1),
                        myz = ops::med(P.M.mu, g, gi, gj + 1, k + 1);
            mm[c] = m0;
            ms[c][0] = ar::mean4(m0, mx, my, mxy);
            const bool harm = FS && k == g.fs - 1;
            ms[c][1] = harm ? ar::harm4(m0, mx, mz, mxz) : ar::mean4(m0, mx, mz, mxz);
            ms[c][2] = harm ? ar::harm4(m0, my, mz, myz) : ar::mean4(m0, my, mz, myz);
        }
        mg[c] = BND == BND_SPONGE ? ar::gain(__ldg(P.B.g[0] + gi), __ldg(P.B.g[1] + gj), __ldg(P.B.g[2] + k)) : 1.0f;
#pragma unroll
        for (int q = 0; q < NFIELD; ++q) sm[q * FCAP + so + c * SP] = __ldcg(P.F.f[q] + go + c * plane);
    }
    // C-PML coefficients of the column; slabs of its cells along z
    const int W = P.B.W;
    const bool psx = BND == BND_CPML && col && (gi < W || gi >= g.nx - W);
    const bool psy = BND == BND_CPML && col && (gj < W || gj >= g.ny - W);
    const float pax = psx ? __ldg(P.B.pa[0] + gi) : 0.f, pbx = psx ? __ldg(P.B.pb[0] + gi) : 0.f;
    const float pay = psy ? __ldg(P.B.pa[1] + gj) : 0.f, pby = psy ? __ldg(P.B.pb[1] + gj) : 0.f;
    const float* paz = P.B.pa[2] + gk;
    const float* pbz = P.B.pb[2] + gk;
    auto psz = [&](int c) { return BND == BND_CPML && (gk + c < W || gk + c >= g.nz - W); };
    float* const ps = sm + NFIELD * FCAP + t;    // PSM: variable q of the thread's cell at ps[q * MAXT]
    if (PSM && nc > 0) {
#pragma unroll
        for (int q = 0; q < 18; ++q)
            if (q < 6 ? psx : q < 12 ? psy : psz(0)) ps[q * MAXT] = P.B.psi[q][go];
    }
    // the thread's halo line
    HaloLine h;
    h.axis = -1;
    {
        const int ax = LY * LZ, ay = LX * LZ, az = LX * LY;
        int e = t, u = 0, v = 0, li = 0;
        auto place = [&](int c) { return c * 18 * P.lines + li; };
        if (e < ax) {
            h.axis = 0;
            li = e;
            u = e % LY; v = e / LY;                                   // j, k
            h.so = (v + 2) * SP + (u + 2) * SX + 2;
            h.go = (k0 + v) * plane + (j0 + u) * g.pitch + i0;
            h.ss = 1; h.gs = 1; h.len = LX;
            h.lo = bi > 0 ? place(cta - 1) : -1;
            h.hi = bi + 1 < P.nbx ? place(cta + 1) : -1;
        } else if ((e -= ax) < ay) {
            h.axis = 1;
            li = P.lcap0 + e;
            u = e % LX; v = e / LX;                                   // i, k
            h.so = (v + 2) * SP + 2 * SX + u + 2;
            h.go = (k0 + v) * plane + j0 * g.pitch + i0 + u;
            h.ss = SX; h.gs = g.pitch; h.len = LY;
            h.lo = bj > 0 ? place(cta - P.nbx) : -1;
            h.hi = bj + 1 < P.nby ? place(cta + P.nbx) : -1;
        } else if ((e -= ay) < az) {
            h.axis = 2;
            li = P.lcap1 + e;
            u = e % LX; v = e / LX;                                   // i, j
            h.so = 2 * SP + (v + 2) * SX + u + 2;
            h.go = k0 * plane + (j0 + v) * g.pitch + i0 + u;
            h.ss = SP; h.gs = plane; h.len = LZ;
            h.lo = bk > 0 ? place(cta - P.nbx * P.nby) : -1;
            h.hi = bk + 1 < P.nbz ? place(cta + P.nbx * P.nby) : -1;
        }
        h.in = place(cta);
    }
    // source taps inside the block
    if (P.S.kind >= 0 && t < P.S.ntap) {
        const Tap& q = P.S.tap[t];
        const int x = q.i - i0, y = q.j - j0, z = q.k - k0;
        const bool in = x >= 0 && x < LX && y >= 0 && y < LY && z >= 0 && z < LZ;
        s_off[t] = in ? q.q * FCAP + (z + 2) * SP + (y + 2) * SX + x + 2 : -1;
        if (in) {
            s_src = 1;
            float b = 1.0f;
            if (P.S.kind == 1) {
                const int c = q.q - VX;
                b = g.cm[2] ? 1.0f / coarse_at(g, 2, q.i + (c == 0 ? 0.5f : 0.0f), q.j + (c == 1 ? 0.5f : 0.0f),
                                               q.k + (c == 2 ? 0.5f : 0.0f))
                            : ops::buoy(P.M, g, c, q.i, q.j, q.k);
            }
            s_amp[t][0] = b;
            s_amp[t][1] = ops::gain(P.B, q.i, q.j, q.k);
        }
    }
    const bool listed = ADJ ? P.sadj != nullptr : P.stage != nullptr;
    const int tl0 = listed ? __ldg(P.tstart + cta) : 0, tl1 = listed ? __ldg(P.tstart + cta + 1) : 0;
    // reverse sweep: accumulators, v^{n+3/2} and the residual's factors
    float acc[ADJ ? CPT : 1][8], vnx[ADJ ? CPT : 1][3];
    if constexpr (ADJ) {
#pragma unroll
        for (int c = 0; c < CPT; ++c)
            if (c < nc) {
#pragma unroll
                for (int q = 0; q < 8; ++q) acc[c][q] = P.A.acc[q][go + c * plane];
                const long long hs = (long long)(P.n0 + P.nsteps - P.h0 + 1) * 3 * P.fstride + go + c * plane;
#pragma unroll
                for (int q = 0; q < 3; ++q) vnx[c][q] = P.vnext ? __ldg(P.vhist + hs + q * P.fstride) : 0.0f;
            }
        for (int x = tl0 + t; x < tl1; x += NT) {
            const Tap q = P.taps[__ldg(P.tlist + x).y];
            P.coef[x] = ops::gain(P.B, q.i, q.j, q.k) * ops::buoy(P.M, g, q.q - VX, q.i, q.j, q.k) * q.w;
        }
    }
    __syncthreads();
    const bool src = s_src != 0;

    // one tap of the source: amplitude of step n into the field's cell
    auto inject = [&](int n, float* hist) {
        if (t < P.S.ntap && s_off[t] >= 0) {
            const Tap& q = P.S.tap[t];
            float amp = __fmul_rn(q.w, __ldg(P.wavelet + n));
            if (P.S.kind == 1) amp = __fmul_rn(amp, s_amp[t][0]);
            amp = __fmul_rn(amp, s_amp[t][1]);
            const float x = __fadd_rn(sm[s_off[t]], amp);
            sm[s_off[t]] = x;
            if (hist) hist[(q.q - VX) * P.fstride + q.k * plane + q.j * g.pitch + q.i] = x;
        }
    };

    // memory variables q0 .. q0 + 2 of one cell: from and to shared memory, or
    // (already fetched) to global memory
    auto psi_get = [&](float* p, int q0) {
        if (PSM)
#pragma unroll
            for (int q = 0; q < 3; ++q) p[q] = ps[(q0 + q) * MAXT];
    };
    auto psi_put = [&](const float* p, int q0, int o) {
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (PSM) ps[(q0 + q) * MAXT] = p[q];
            else P.B.psi[q0 + q][o] = p[q];
    };

    float* vcap = P.vcap;
    for (int m = 0; m < P.nsteps; ++m) {
        const int n = ADJ ? P.n0 + P.nsteps - 1 - m : P.n0 + m;
        // opaque to the compiler, so that addresses derived from these are
        // formed where they are used and not kept (spilled) across steps
        asm volatile("" : "+r"(h.in), "+r"(h.lo), "+r"(h.hi), "+r"(h.so), "+r"(h.axis));
        // ---- velocity phase ----
        float px[CPT][3], py[CPT][3], pz[CPT][3];
        if (BND == BND_CPML && !PSM) {           // memory variables, fetched before the wait
#pragma unroll
            for (int c = 0; c < CPT; ++c)
                if (c < nc) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (psx) px[c][q] = P.B.psi[q][go + c * plane];
                        if (psy) py[c][q] = P.B.psi[6 + q][go + c * plane];
                        if (psz(c)) pz[c][q] = P.B.psi[12 + q][go + c * plane];
                    }
                }
        }
        // reverse sweep: the history of this step, read before the wait (own
        // cells, and the layers its strain rates reach across the faces)
        float hv[ADJ ? CPT : 1][3], hl[ADJ ? 9 : 1];
        if constexpr (ADJ) {
            const float* hist = P.vhist + (long long)(n - P.h0 + 1) * 3 * P.fstride;
#pragma unroll
            for (int c = 0; c < CPT; ++c)
                if (c < nc)
#pragma unroll
                    for (int q = 0; q < 3; ++q) hv[c][q] = __ldg(hist + q * P.fstride + go + c * plane);
            if (h.axis >= 0) {
                int q[3];
                line_fields<false>(h.axis, q);
#pragma unroll
                for (int e = 0; e < 9; ++e) {
                    const bool dp = e >= 3, hi = dp ? from_hi<true>(e % 3) : from_hi<false>(e % 3);
                    const int at = dp ? layer_at<true>(h, e % 3) : layer_at<false>(h, e % 3);
                    if ((hi ? h.hi : h.lo) >= 0) hl[e] = __ldg(hist + q[e / 3] * P.fstride + h.go + at * h.gs);
                }
            }
        }
        bool ok = true;
        if (m > 0) ok = halo_recv<true, FCAP>(h, P, sm, P.epoch + m);
        else halo_first<true, FCAP>(h, P, sm);
        if constexpr (ADJ) {
#pragma unroll
            for (int c = 0; c < CPT; ++c)
                if (c < nc)
#pragma unroll
                    for (int q = 0; q < 3; ++q) sm[(H0 + q) * FCAP + so + c * SP] = hv[c][q];
            if (h.axis >= 0) {
                int q[3];
                line_fields<false>(h.axis, q);
#pragma unroll
                for (int e = 0; e < 9; ++e) {
                    const bool dp = e >= 3, hi = dp ? from_hi<true>(e % 3) : from_hi<false>(e % 3);
                    const int at = dp ? layer_at<true>(h, e % 3) : layer_at<false>(h, e % 3);
                    if ((hi ? h.hi : h.lo) >= 0) sm[(H0 + q[e / 3]) * FCAP + h.so + at * h.ss] = hl[e];
                }
            }
        }
        if (__syncthreads_or(!ok)) return;
        if (nc > 0) {
            const float* s = sm + so;
            float v[CPT][3];
            float zz[CPT + 3], xz[CPT + 3], yz[CPT + 3];     // szz from k-1, sxz / syz from k-2
#pragma unroll
            for (int c = 0; c < CPT + 3; ++c) {
                zz[c] = s[SZZ * FCAP + (c - 1) * SP];
                xz[c] = s[SXZ * FCAP + (c - 2) * SP];
                yz[c] = s[SYZ * FCAP + (c - 2) * SP];
            }
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const float* xx = s + SXX * FCAP + c * SP;
                const float* yy = s + SYY * FCAP + c * SP;
                const float* xy = s + SXY * FCAP + c * SP;
                const float* fxz = s + SXZ * FCAP + c * SP;
                const float* fyz = s + SYZ * FCAP + c * SP;
                const ZW zw = zweights<FS ? ZS_FWD : ZS_NONE>(g, gk + c);
                const ZT zt{};
                constexpr int ZF = FS ? ZS_FWD : ZS_NONE;
                float dxx = ar::d4(g.c1x, g.c2x, xx[-1], s[SXX * FCAP + c * SP], xx[1], xx[2]);
                float dxy = ar::d4(g.c1y, g.c2y, xy[-2 * SX], xy[-SX], s[SXY * FCAP + c * SP], xy[SX]);
                float dxz = zdiff<ZF, false>(g, zw, zt, xz[c], xz[c + 1], xz[c + 2], xz[c + 3]);
                float dyx = ar::d4(g.c1x, g.c2x, xy[-2], xy[-1], s[SXY * FCAP + c * SP], xy[1]);
                float dyy = ar::d4(g.c1y, g.c2y, yy[-SX], s[SYY * FCAP + c * SP], yy[SX], yy[2 * SX]);
                float dyz = zdiff<ZF, false>(g, zw, zt, yz[c], yz[c + 1], yz[c + 2], yz[c + 3]);
                float dzx = ar::d4(g.c1x, g.c2x, fxz[-2], fxz[-1], s[SXZ * FCAP + c * SP], fxz[1]);
                float dzy = ar::d4(g.c1y, g.c2y, fyz[-2 * SX], fyz[-SX], s[SYZ * FCAP + c * SP], fyz[SX]);
                float dzz = zdiff<ZF, true>(g, zw, zt, zz[c], zz[c + 1], zz[c + 2], zz[c + 3]);
                if (BND == BND_CPML && c < nc) {
                    const int o = go + c * plane;
                    if (psx) {
                        psi_get(px[c], 0);
                        ar::pml(px[c][0], pax, pbx, dxx); ar::pml(px[c][1], pax, pbx, dyx); ar::pml(px[c][2], pax, pbx, dzx);
                        psi_put(px[c], 0, o);
                    }
                    if (psy) {
                        psi_get(py[c], 6);
                        ar::pml(py[c][0], pay, pby, dxy); ar::pml(py[c][1], pay, pby, dyy); ar::pml(py[c][2], pay, pby, dzy);
                        psi_put(py[c], 6, o);
                    }
                    if (psz(c)) {
                        psi_get(pz[c], 12);
                        const float a = __ldg(paz + c), b = __ldg(pbz + c);
                        ar::pml(pz[c][0], a, b, dxz); ar::pml(pz[c][1], a, b, dyz); ar::pml(pz[c][2], a, b, dzz);
                        psi_put(pz[c], 12, o);
                    }
                }
                if constexpr (ADJ) {
                    // gradient products of this reverse step (see k_velocity, M_GRAD)
                    const float* hx = s + H0 * FCAP + c * SP;
                    const float* hy = hx + FCAP;
                    const float* hz = hy + FCAP;
                    const float ex = ar::d4(g.c1x, g.c2x, hx[-2], hx[-1], hx[0], hx[1]);
                    const float ey = ar::d4(g.c1y, g.c2y, hy[-2 * SX], hy[-SX], hy[0], hy[SX]);
                    const float ez = ar::d4(g.c1z, g.c2z, hz[-2 * SP], hz[-SP], hz[0], hz[SP]);
                    const float gxy = ar::d4(g.c1y, g.c2y, hx[-SX], hx[0], hx[SX], hx[2 * SX]) +
                                      ar::d4(g.c1x, g.c2x, hy[-1], hy[0], hy[1], hy[2]);
                    const float gxz = ar::d4(g.c1z, g.c2z, hx[-SP], hx[0], hx[SP], hx[2 * SP]) +
                                      ar::d4(g.c1x, g.c2x, hz[-1], hz[0], hz[1], hz[2]);
                    const float gyz = ar::d4(g.c1z, g.c2z, hy[-SP], hy[0], hy[SP], hy[2 * SP]) +
                                      ar::d4(g.c1y, g.c2y, hz[-SX], hz[0], hz[SX], hz[2 * SX]);
                    const float ux = s[SXX * FCAP + c * SP], uy = s[SYY * FCAP + c * SP], uz = s[SZZ * FCAP + c * SP];
                    acc[c][0] += P.gdt * (ex + ey + ez) * (ux + uy + uz);
                    acc[c][1] += P.gdt * (ex * ux + ey * uy + ez * uz);
                    acc[c][2] += P.gdt * gxy * s[SXY * FCAP + c * SP];
                    acc[c][3] += P.gdt * gxz * s[SXZ * FCAP + c * SP];
                    acc[c][4] += P.gdt * gyz * s[SYZ * FCAP + c * SP];
                    if (m > 0 || P.vnext) {
                        const float iG = 1.0f / mg[c];
                        acc[c][5] += (vnx[c][0] * iG - hx[0]) * s[VX * FCAP + c * SP];
                        acc[c][6] += (vnx[c][1] * iG - hy[0]) * s[VY * FCAP + c * SP];
                        acc[c][7] += (vnx[c][2] * iG - hz[0]) * s[VZ * FCAP + c * SP];
                    }
                    vnx[c][0] = hx[0];
                    vnx[c][1] = hy[0];
                    vnx[c][2] = hz[0];
                }
                v[c][0] = ar::vnew(s[VX * FCAP + c * SP], P.dt, mb[c][0], dxx, dxy, dxz);
                v[c][1] = ar::vnew(s[VY * FCAP + c * SP], P.dt, mb[c][1], dyx, dyy, dyz);
                v[c][2] = ar::vnew(s[VZ * FCAP + c * SP], P.dt, mb[c][2], dzx, dzy, dzz);
            }
#pragma unroll
            for (int c = 0; c < CPT; ++c)
                if (c < nc) {
                    const int o = go + c * plane;
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        const float x = BND == BND_SPONGE ? __fmul_rn(v[c][q], mg[c]) : v[c][q];
                        sm[(VX + q) * FCAP + so + c * SP] = x;
                        if (vcap) vcap[q * P.fstride + o] = x;
                    }
                }
        }
        if (src && P.S.kind == 1) {
            __syncthreads();
            inject(n, vcap);
        }
        if (ADJ && tl1 > tl0) {                  // residual of step n (taps may share a cell)
            __syncthreads();
            for (int x = tl0 + t; x < tl1; x += NT) {
                const int2 e = __ldg(P.tlist + x);
                atomicAdd(sm + e.x, P.coef[x] * __ldg(P.sadj + (long long)(e.y >> 3) * P.ld + n));
            }
        }
        __syncthreads();
        halo_send<false, FCAP>(h, P, sm, P.epoch + m + 1);
        if (vcap) vcap += 3 * P.fstride;
        // v^{n+1/2} at the receiver taps of this block
        if (!ADJ)
            for (int x = tl0 + t; x < tl1; x += NT) {
                const int2 e = __ldg(P.tlist + x);
                P.stage[(size_t)m * P.ntap + e.y] = sm[e.x];
            }
        // ---- stress phase ----
        asm volatile("" : "+r"(h.in), "+r"(h.lo), "+r"(h.hi), "+r"(h.so), "+r"(h.axis));
        if (BND == BND_CPML && !PSM) {
#pragma unroll
            for (int c = 0; c < CPT; ++c)
                if (c < nc) {
#pragma unroll
                    for (int q = 0; q < 3; ++q) {
                        if (psx) px[c][q] = P.B.psi[3 + q][go + c * plane];
                        if (psy) py[c][q] = P.B.psi[9 + q][go + c * plane];
                        if (psz(c)) pz[c][q] = P.B.psi[15 + q][go + c * plane];
                    }
                }
        }
        ok = halo_recv<false, FCAP>(h, P, sm, P.epoch + m + 1);
        if (__syncthreads_or(!ok)) return;
        if (nc > 0) {
            const float* s = sm + so;
            float r[CPT][6];
            float zx[CPT + 3], zy[CPT + 3], zv[CPT + 3];     // vx / vy from k-1, vz from k-2
#pragma unroll
            for (int c = 0; c < CPT + 3; ++c) {
                zx[c] = s[VX * FCAP + (c - 1) * SP];
                zy[c] = s[VY * FCAP + (c - 1) * SP];
                zv[c] = s[VZ * FCAP + (c - 2) * SP];
            }
#pragma unroll
            for (int c = 0; c < CPT; ++c) {
                const float* vx = s + VX * FCAP + c * SP;
                const float* vy = s + VY * FCAP + c * SP;
                const float* vz = s + VZ * FCAP + c * SP;
                const ZW zw = zweights<FS ? ZS_FWD : ZS_NONE>(g, gk + c);
                const ZT zt{};
                constexpr int ZF = FS ? ZS_FWD : ZS_NONE;
                float exx = ar::d4(g.c1x, g.c2x, vx[-2], vx[-1], s[VX * FCAP + c * SP], vx[1]);
                float eyy = ar::d4(g.c1y, g.c2y, vy[-2 * SX], vy[-SX], s[VY * FCAP + c * SP], vy[SX]);
                float ezz = zdiff<ZF, false>(g, zw, zt, zv[c], zv[c + 1], zv[c + 2], zv[c + 3]);
                float vxy = ar::d4(g.c1y, g.c2y, vx[-SX], s[VX * FCAP + c * SP], vx[SX], vx[2 * SX]);
                float vyx = ar::d4(g.c1x, g.c2x, vy[-1], s[VY * FCAP + c * SP], vy[1], vy[2]);
                float vxz = zdiff<ZF, true>(g, zw, zt, zx[c], zx[c + 1], zx[c + 2], zx[c + 3]);
                float vzx = ar::d4(g.c1x, g.c2x, vz[-1], s[VZ * FCAP + c * SP], vz[1], vz[2]);
                float vyz = zdiff<ZF, true>(g, zw, zt, zy[c], zy[c + 1], zy[c + 2], zy[c + 3]);
                float vzy = ar::d4(g.c1y, g.c2y, vz[-SX], s[VZ * FCAP + c * SP], vz[SX], vz[2 * SX]);
                if (BND == BND_CPML && c < nc) {
                    const int o = go + c * plane;
                    if (psx) {
                        psi_get(px[c], 3);
                        ar::pml(px[c][0], pax, pbx, exx); ar::pml(px[c][1], pax, pbx, vyx); ar::pml(px[c][2], pax, pbx, vzx);
                        psi_put(px[c], 3, o);
                    }
                    if (psy) {
                        psi_get(py[c], 9);
                        ar::pml(py[c][0], pay, pby, eyy); ar::pml(py[c][1], pay, pby, vxy); ar::pml(py[c][2], pay, pby, vzy);
                        psi_put(py[c], 9, o);
                    }
                    if (psz(c)) {
                        psi_get(pz[c], 15);
                        const float a = __ldg(paz + c), b = __ldg(pbz + c);
                        ar::pml(pz[c][0], a, b, ezz); ar::pml(pz[c][1], a, b, vxz); ar::pml(pz[c][2], a, b, vyz);
                        psi_put(pz[c], 15, o);
                    }
                }
                const float l2m = ar::l2m(ml[c], mm[c]);
                r[c][0] = ar::snormal(s[SXX * FCAP + c * SP], P.dt, l2m, ml[c], exx, eyy, ezz);
                r[c][1] = ar::snormal(s[SYY * FCAP + c * SP], P.dt, l2m, ml[c], eyy, exx, ezz);
                r[c][2] = ar::snormal(s[SZZ * FCAP + c * SP], P.dt, l2m, ml[c], ezz, exx, eyy);
                r[c][3] = ar::sshear(s[SXY * FCAP + c * SP], P.dt, ms[c][0], vxy, vyx);
                r[c][4] = ar::sshear(s[SXZ * FCAP + c * SP], P.dt, ms[c][1], vxz, vzx);
                r[c][5] = ar::sshear(s[SYZ * FCAP + c * SP], P.dt, ms[c][2], vyz, vzy);
            }
#pragma unroll
            for (int c = 0; c < CPT; ++c)
                if (c < nc) {
#pragma unroll
                    for (int q = 0; q < 6; ++q) {
                        const float x = BND == BND_SPONGE ? __fmul_rn(r[c][q], mg[c]) : r[c][q];
                        sm[(SXX + q) * FCAP + so + c * SP] = x;
                    }
                }
        }
        if (src && P.S.kind == 0) {
            __syncthreads();
            inject(n, nullptr);
        }
        __syncthreads();
        if (m + 1 < P.nsteps) halo_send<true, FCAP>(h, P, sm, P.epoch + m + 1);
        if constexpr (ADJ)
            if (n > P.h0 && (n - P.h0) % P.flush == 0) {
#pragma unroll
                for (int c = 0; c < CPT; ++c)
                    if (c < nc)
#pragma unroll
                        for (int q = 0; q < 8; ++q) {
                            P.A.acc64[q][go + c * plane] += (double)acc[c][q];
                            acc[c][q] = 0.0f;
                        }
            }
    }
    if constexpr (ADJ)
#pragma unroll
        for (int c = 0; c < CPT; ++c)
            if (c < nc)
#pragma unroll
                for (int q = 0; q < 8; ++q) P.A.acc[q][go + c * plane] = acc[c][q];
#pragma unroll
    for (int c = 0; c < CPT; ++c)
        if (c < nc)
#pragma unroll
            for (int q = 0; q < NFIELD; ++q) P.F.f[q][go + c * plane] = sm[q * FCAP + so + c * SP];
    if (PSM && nc > 0) {
#pragma unroll
        for (int q = 0; q < 18; ++q)
            if (q < 6 ? psx : q < 12 ? psy : psz(0)) P.B.psi[q][go] = ps[q * MAXT];
    }
}

// Receiver samples of the steps of a resident launch from the staged tap
// values: one thread per (sample row, step), 8 taps in the order of
// ops::record_one; a non-finite sample sets bit 16 of *err.
__global__ void k_resident_record(const float* __restrict__ stage, int ntap,
                                  const Tap* __restrict__ taps, int rows, int nsteps,
                                  float* __restrict__ seis, int ld, int n0, int* err) {
    const int x = blockIdx.x * blockDim.x + threadIdx.x;
    if (x >= rows * nsteps) return;
    const int t = x % rows, m = x / rows;
    const float* s = stage + (size_t)m * ntap + 8 * t;
    float acc = 0.0f;
#pragma unroll
    for (int q = 0; q < 8; ++q) acc = __fmaf_rn(taps[8 * t + q].w, s[q], acc);
    if (!isfinite(acc)) atomicOr(err, 16);
    seis[(long long)t * ld + n0 + m] = acc;
}

using Kern = void (*)(ResParams);
template <int CPT, int MAXT>
Kern pick(int bnd, bool fs) {
    switch (bnd) {
        case BND_SPONGE: return fs ? k_resident<BND_SPONGE, 1, CPT, MAXT> : k_resident<BND_SPONGE, 0, CPT, MAXT>;
        case BND_CPML:
            if constexpr (MAXT != 768)           // resident_plan: at most 8 planes
                return fs ? k_resident<BND_CPML, 1, CPT, MAXT> : k_resident<BND_CPML, 0, CPT, MAXT>;
            return nullptr;
        default: return fs ? k_resident<BND_NONE, 1, CPT, MAXT> : k_resident<BND_NONE, 0, CPT, MAXT>;
    }
}
// Cells per thread along z: one z-group of COLS threads per CPT planes.
// Blocks of at most 4 planes take a thread per cell (32^3: 4.6 us a step),
// larger ones 4 cells per thread, whose shared columns save loads (64^3 in
// blocks of 8 planes: 5.9 us, 6.7 with two cells on 1024 threads; a thread's
// own field values kept in registers as well gained nothing).  Every choice has
// at least as many threads as halo lines.
int cells_per_thread(int lz) { return lz <= 4 ? 1 : 4; }
int block_threads(int lz) {
    const int cpt = cells_per_thread(lz);
    return COLS * std::max(2, (lz + cpt - 1) / cpt);
}
Kern kernel_for(int bnd, bool fs, int lz) {
    return lz <= 4 ? pick<1, 1024>(bnd, fs) : lz <= 8 ? pick<4, 512>(bnd, fs) : pick<4, 768>(bnd, fs);
}
size_t smem_bytes(int bnd, int lz, bool adj) {
    const size_t f = (size_t)(NFIELD + (adj ? 3 : 0)) * fcap(lz);
    return (f + (bnd == BND_CPML && lz <= 4 ? 18 * 1024 : 0)) * sizeof(float);
}
// Reverse sweep: blocks of at most 8 planes, no C-PML, no free surface.
Kern adjoint_kernel(int bnd, int lz) {
    if (lz > 8 || bnd == BND_CPML) return nullptr;
    if (lz <= 4)
        return bnd == BND_SPONGE ? k_resident<BND_SPONGE, 0, 1, 1024, true> : k_resident<BND_NONE, 0, 1, 1024, true>;
    return bnd == BND_SPONGE ? k_resident<BND_SPONGE, 0, 4, 512, true> : k_resident<BND_NONE, 0, 4, 512, true>;
}

}  // namespace

// A grid whose blocks fit: the block counts per axis, chosen among all with
// at most one CTA per SM to minimise the cells and halo cells of a CTA (a
// half-warp covers one row of up to 16 cells whatever its length, a thread of
// a block of more than 4 planes 4 of them; blocks of more than 8 planes need
// 768 threads, whose 80 registers spill: 64^3 in blocks of 8 planes 5.9 us a
// step, in blocks of 11 planes 7.7; with C-PML, blocks of more than 4 planes
// leave the memory variables in global memory: 70 x 45 x 37 in blocks of 8
// planes 9.9 us).
bool resident_plan(const DevGrid& g, int bnd, int sms, ResidentPlan* out) {
    if ((long long)g.nx * g.ny * g.nz > (long long)sms * MX * MY * MAXZ) return false;
    const int maxz = bnd == BND_CPML ? 8 : MAXZ;     // registers of the memory variables
    long long best = -1;
    for (int bx = (g.nx + MX - 1) / MX; bx <= std::max(1, g.nx / 2) && bx <= sms; ++bx)
        for (int by = (g.ny + MY - 1) / MY; by <= std::max(1, g.ny / 2) && bx * by <= sms; ++by)
            for (int bz = (g.nz + maxz - 1) / maxz; bz <= std::max(1, g.nz / 2) && bx * by * bz <= sms; ++bz) {
                const long long lx = (g.nx + bx - 1) / bx, ly = (g.ny + by - 1) / by, lz = (g.nz + bz - 1) / bz;
                const long long cells = MX * ly * (lz <= 4 ? lz : lz <= 8 ? (bnd == BND_CPML ? 16 : 8) : 16);
                const long long cost = cells + 3 * (ly * lz + lx * lz + lx * ly);
                if (best < 0 || cost < best) {
                    best = cost;
                    out->nbx = bx; out->nby = by; out->nbz = bz;
                    out->lz = (int)lz;
                    out->lines[0] = (int)(ly * lz);
                    out->lines[1] = (int)(lx * lz);
                    out->lines[2] = (int)(lx * ly);
                }
            }
    return best >= 0;
}

size_t resident_inbox_bytes(const ResidentPlan& p) {
    return (size_t)p.nbx * p.nby * p.nbz * 2 * 9 * (p.lines[0] + p.lines[1] + p.lines[2]) *
           sizeof(unsigned long long);
}

// The taps of each CTA's block: start[c] .. start[c + 1] of list holds
// (shared-memory offset, tap index) pairs.
void resident_taps(const ResidentPlan& p, const DevGrid& g, const Tap* taps, int ntap,
                   std::vector<int2>* list, std::vector<int>* start) {
    auto block_of = [](int n, int nb, int x) {
        int b = (int)((long long)x * nb / n);
        while (b + 1 < nb && block_lo(n, nb, b + 1) <= x) ++b;
        while (b > 0 && block_lo(n, nb, b) > x) --b;
        return b;
    };
    const int nc = p.nbx * p.nby * p.nbz;
    std::vector<int> cta(ntap);
    start->assign(nc + 1, 0);
    for (int t = 0; t < ntap; ++t) {
        const int x = block_of(g.nx, p.nbx, taps[t].i), y = block_of(g.ny, p.nby, taps[t].j),
                  z = block_of(g.nz, p.nbz, taps[t].k);
        cta[t] = (z * p.nby + y) * p.nbx + x;
        ++(*start)[cta[t] + 1];
    }
    for (int c = 0; c < nc; ++c) (*start)[c + 1] += (*start)[c];
    std::vector<int> at(start->begin(), start->end() - 1);
    list->resize(ntap);
    for (int t = 0; t < ntap; ++t) {
        const Tap& q = taps[t];
        const int c = cta[t];
        const int x = q.i - block_lo(g.nx, p.nbx, c % p.nbx), y = q.j - block_lo(g.ny, p.nby, (c / p.nbx) % p.nby),
                  z = q.k - block_lo(g.nz, p.nbz, c / (p.nbx * p.nby));
        (*list)[at[c]++] = make_int2(q.q * fcap(p.lz) + (z + 2) * SP + (y + 2) * SX + x + 2, t);
    }
}

cudaError_t resident_prepare(const ResidentPlan& p, int bnd) {
    const Kern ks[3] = {kernel_for(bnd, false, p.lz), kernel_for(bnd, true, p.lz), adjoint_kernel(bnd, p.lz)};
    for (int v = 0; v < 3; ++v) {
        if (!ks[v]) continue;
        const size_t smem = smem_bytes(bnd, p.lz, v == 2);
        int occ = 0;
        cudaError_t e = cudaFuncSetAttribute(ks[v], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, ks[v], block_threads(p.lz), smem);
        if (e != cudaSuccess) return e;
        if (occ < 1) return cudaErrorInvalidConfiguration;
    }
    return cudaSuccess;
}

bool resident_adjoint_supported(const ResidentPlan& p, const DevGrid& g, int bnd) {
    return adjoint_kernel(bnd, p.lz) != nullptr && g.fs == kNoSurface && !g.cm[0];
}

namespace {
ResParams res_params(const ResidentRun& r) {
    const ResidentPlan& p = *r.plan;
    ResParams P{};
    P.g = r.g;
    P.F = r.F;
    P.M = r.M;
    P.B = r.B;
    P.dt = r.dt;
    P.S.kind = -1;
    P.n0 = r.n0;
    P.nsteps = r.nsteps;
    P.inbox = r.inbox;
    P.epoch = r.epoch;
    P.lcap0 = p.lines[0];
    P.lcap1 = p.lines[0] + p.lines[1];
    P.lines = P.lcap1 + p.lines[2];
    P.err = r.err;
    P.nbx = p.nbx;
    P.nby = p.nby;
    P.nbz = p.nbz;
    P.tlist = r.tlist;
    P.tstart = r.tstart;
    P.ntap = 24 * r.nrec;
    P.fstride = r.fstride;
    P.wait_ns = r.test_wait_ms > 0 ? r.test_wait_ms * 1000000ull : 2000000000ull;   // 2 s per wait
    P.mute = r.test_wait_ms > 0 ? 0 : -1;
    return P;
}
}  // namespace

// Reverse steps n0 + nsteps - 1 .. n0 of one resident history range.
cudaError_t launch_resident_adjoint(const ResidentRun& r, const ResidentAdjoint& a, cudaStream_t st) {
    const ResidentPlan& p = *r.plan;
    ResParams P = res_params(r);
    P.vhist = a.vhist;
    P.h0 = a.h0;
    P.vnext = a.vnext;
    P.flush = a.flush;
    P.A = a.A;
    P.gdt = a.gdt;
    P.sadj = r.nrec > 0 ? a.sadj : nullptr;
    P.ld = r.ld;
    P.taps = r.taps;
    P.coef = r.stage;
    void* args[] = {&P};
    return cudaLaunchCooperativeKernel((const void*)adjoint_kernel(r.B.kind, p.lz), dim3(p.nbx * p.nby * p.nbz),
                                       dim3(block_threads(p.lz)), args, smem_bytes(r.B.kind, p.lz, true), st);
}

// Measured (GB300, us per step, without / with C-PML), against the replayed
// graph of the passes: 32^3 4.6 / 4.7 (10.0 / 15.4), 70 x 45 x 37 4.8 / 6.1
// (11.9 / 18.3), 64^3 5.8 / 10.0 (11.9 / 17.8), 80 x 80 x 70 7.8 (17.9).  Of
// the 2 us a phase takes at 32^3, most is the exchange (store to another SM's
// poll) and the two barriers around it; at 64^3 the shared-memory loads of the
// update (29 to 38 words a cell) take half.
cudaError_t launch_resident(const ResidentRun& r, cudaStream_t st) {
    const ResidentPlan& p = *r.plan;
    ResParams P = res_params(r);
    P.S = *r.S;
    P.wavelet = r.wavelet;
    P.stage = r.seis ? r.stage : nullptr;
    P.vcap = r.vcap;
    const Kern k = kernel_for(r.B.kind, r.g.fs != kNoSurface, p.lz);
    const dim3 grid(p.nbx * p.nby * p.nbz), blk(block_threads(p.lz));
    void* args[] = {&P};
    cudaError_t e = cudaLaunchCooperativeKernel((const void*)k, grid, blk, args, smem_bytes(r.B.kind, p.lz, false), st);
    if (e != cudaSuccess || !P.stage) return e;
    const int rows = 3 * r.nrec;
    const long long n = (long long)rows * r.nsteps;
    k_resident_record<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(
        r.stage, P.ntap, r.taps, rows, r.nsteps, r.seis, r.ld, r.n0, r.err);
    return cudaGetLastError();
}

}  // namespace ews
