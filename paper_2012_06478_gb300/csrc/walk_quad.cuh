// walk_quad.cuh -- the plain form's time step (elastic collision, no absorbing
// membranes) with four lanes to a walker, for runs of too few walkers to fill
// the GPU with one thread each.
//
// What bounds a small run: the step's dependent chain, not the arithmetic
// units.  In the one-thread kernel a warp's step is some 2500 instructions --
// the integer-ALU arithmetic of three axes, one after the other -- and with a
// warp or two on each scheduler nothing hides their latency.  Here lane a of a
// walker's four has axis a: its offset, displacement, face time and phases, so
// that an axis' division and products are done once for all three.  The step's
// direction depends on no state, so each lane draws one of the next four
// steps' and the four share them through shared memory.  A warp holds 8
// walkers instead of 32, which also leaves fewer face events to wait for.
// Every operation on a walker's numbers is the one-thread kernel's, in its
// order: the same bits.
//
// 600 steps of 1e4 walkers on 64^3 axons, the call: 1.72 ms against 2.95 (one warp
// on each of 313 schedulers there; here two on each).  Seven blocks an SM (72
// registers) rather than five: 2.62 ms against 3.15 for 28 000 walkers, 2.95 against
// 3.35 for 32 000, and 1.72 against 1.69 for 1e4.  Several waveforms have no bound.
#pragma once

#include "walk_kernel.cuh"

namespace rms {

constexpr int kQuadWalkers = 32;  // walkers of a block of kWalkBlock threads: a warp of the one-thread kernel

template <int NS, int RELAX, bool SANE>
__global__ void __launch_bounds__(kWalkBlock, NS == 1 ? 7 : 0)
walk_quad_kernel(Geometry g, Tables<double> t, WalkerState<double> st, RunCtl ctl, int64_t k_begin, int64_t k_end,
                 int32_t rec)
{
    constexpr double kZero = 0.0;
    const double kInf = __longlong_as_double(0x7FF0000000000000LL);
    __shared__ int32_t s_cancel;
    __shared__ double s_n[kWalkBlock][4];   // a lane's direction; its last two words (membrane events)
    __shared__ double s_mom[kQuadWalkers][4];
    __shared__ double s_red[kMoments];
    if (threadIdx.x == 0) s_cancel = ctl.cancel ? *ctl.cancel : 0;
    __syncthreads();
    if (s_cancel) return;

    uint32_t rk[kRoundKeys];
#pragma unroll
    for (int i = 0; i < kRoundKeys; ++i) rk[i] = ctl.rk[i];
    const int ax = threadIdx.x & 3, a = ax < 3 ? ax : 2;  // lane 3 copies axis 2 without its events
    const int quad = threadIdx.x & 28;                    // the walker's first lane in the warp
    const int64_t slot = (int64_t)blockIdx.x * kQuadWalkers + (threadIdx.x >> 2);
    const bool active = slot < ctl.n_walkers;  // beyond the last walker: a copy of it that writes nothing
    const int64_t li = active ? slot : ctl.n_walkers - 1;
    const uint64_t w = (uint64_t)(ctl.w_begin + (st.wid ? (int64_t)st.wid[li] : li));
    const int32_t sy = g.nx, sz = g.nx * g.ny;
    const int32_t L = t.n_labels;
    const bool relax = RELAX != 0;
    const double lp = g.voxel_um;

    const auto of_axis = [a](auto x, auto y, auto z) { return a == 0 ? x : (a == 1 ? y : z); };
    double o = of_axis(st.o[0], st.o[1], st.o[2])[li];
    const double o0 = of_axis(st.o0[0], st.o0[1], st.o0[2])[li];
    int32_t di = of_axis(st.di[0], st.di[1], st.di[2])[li];
    int32_t v = wrapped(st.i0[0][li] + st.di[0][li], g.nx) + sy * wrapped(st.i0[1][li] + st.di[1][li], g.ny) +
                sz * wrapped(st.i0[2][li] + st.di[2][li], g.nz);
    uint32_t fm = __ldg(g.faces + v);
    int32_t c = st.c[li];
    double sc = __ldg(t.s + c);
    double A = st.A[li];
    double ph[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) ph[s] = s < ctl.n_shapes ? st.phase[((int64_t)s * 3 + a) * ctl.n_walkers + li] : kZero;
    int32_t next_rec = rec < ctl.n_rec ? __ldg(t.rec_step + rec) : INT32_MAX;
    __syncthreads();  // the copies of the last walker have read it before its own lanes write it back

    for (int32_t k = (int32_t)k_begin + 1; k <= (int32_t)k_end; ++k) {
        double wg = kZero;
        bool graded;
        if constexpr (NS == 1) {
            wg = __ldg(t.wG + (k - 1));
            graded = nonzero(wg);
        } else {
            graded = (__ldg(t.flags + (k - 1)) & 1u) != 0u;
        }
        int mode = 0;
        if (relax) mode = t.mode ? (int)__ldg(t.mode + (k - 1)) : 0;
        // ---- directions of the next four steps, one a lane
        const int turn = (k - (int32_t)k_begin - 1) & 3;
        if (turn == 0) {
            const U4 x = philox4x32_10_rk(
                U4{(uint32_t)w, (uint32_t)(w >> 32), (uint32_t)(k + ax), kTagDir << 16}, rk);
            double n3[3];
            direction_from<true>(x.x, x.y, t.trig, n3);
            __syncwarp();
            s_n[threadIdx.x][0] = n3[0];
            s_n[threadIdx.x][1] = n3[1];
            s_n[threadIdx.x][2] = n3[2];
            s_n[threadIdx.x][3] = __hiloint2double((int)x.w, (int)x.z);
            __syncwarp();
        }
        const double *from = s_n[(threadIdx.x & ~3) + turn];
        double n = from[a];
        double rate = kZero;
        if (relax) rate = __ldg(t.dtR + mode * L + c);
        double d = times_nz<SANE>(n, sc);
        double T = kInf;
        if (ax < 3 && (SANE || dgt0(d) || dlt0(d)))
            T = over<SANE>(dgt0(d) ? 1.0 - o : o, __longlong_as_double(dbits(d) & 0x7FFFFFFFFFFFFFFFLL));
        double tau = kZero;
#pragma unroll 1
        for (int ev = 0; ev < 3; ++ev) {
            // the earliest face time of the walker's axes, ties to the lower axis
            long long tb = dbits(T);
            {
                const long long p1 = __shfl_xor_sync(0xffffffffu, tb, 1);
                tb = p1 < tb ? p1 : tb;
                const long long p2 = __shfl_xor_sync(0xffffffffu, tb, 2);
                tb = p2 < tb ? p2 : tb;
            }
            const double tmin = __longlong_as_double(tb);
            const bool event = dlt_nn(tmin, 1.0);
            if (!__any_sync(0xffffffffu, event)) break;
            const uint32_t at = __ballot_sync(0xffffffffu, dbits(T) == tb) >> quad;
            const uint32_t ups = __ballot_sync(0xffffffffu, dgt0(d)) >> quad;
            if (event) {
                const int best = __ffs((int)(at & 7u)) - 1;
                const bool up = ((ups >> best) & 1u) != 0u, mine = ax == best;
                const double dts = tmin - tau;
                if (relax) A = A + times_any<SANE>(dts, rate);
                tau = tmin;
                if (mine) {
                    T = kInf;
                    o = up ? 0.0 : 1.0;
                    di += up ? 1 : -1;
                } else {
                    o = dclamp01(o + times<SANE>(dts, d));
                }
                const int32_t sb = best == 2 ? sz : (best == 1 ? sy : 1);
                const uint32_t bit = (best == 2 ? kFaceZ : (best == 1 ? kFaceY : kFaceX)) << (up ? 3 : 0);
                int32_t nv = up ? v + sb : v - sb;
                if (!(fm & bit)) {  // not the same label inside the volume: a membrane, or the volume's edge
                    if (fm & kFaceEdge)
                        nv = edge_voxel(v, nv, best, up, g.nx, g.ny, g.nz, g.div_x, g.div_xy, g.periodic);
                    const int32_t c2 = nv < 0 ? -1 : (int32_t)__ldg(g.labels + nv);
                    if (c2 != c) {
                        const uint32_t P = c2 < 0 ? 0u : __ldg(t.T + (int64_t)c * L + c2);
                        bool cross = false;
                        if (P != 0u) {
                            const uint32_t word = ev == 0   ? (uint32_t)__double2loint(from[3])
                                                  : ev == 1 ? (uint32_t)__double2hiint(from[3])
                                                            : perm_word(ctl.seed, w, (uint32_t)k, 0u);
                            cross = word < P;
                        }
                        if (cross) {
                            c = c2;
                            if (relax) rate = __ldg(t.dtR + mode * L + c);
                            const double sn = __ldg(t.s + c);
                            if (dbits(sn) != dbits(sc)) {
                                sc = sn;
                                d = times_nz<SANE>(n, sc);
                                if (dbits(T) != 0x7FF0000000000000LL)
                                    T = tau + over<SANE>(dgt0(d) ? 1.0 - o : o,
                                                      __longlong_as_double(dbits(d) & 0x7FFFFFFFFFFFFFFFLL));
                            }
                        } else {  // reflected: stays in its voxel, at the face
                            nv = v;
                            if (mine) {
                                n = dneg(n);
                                d = dneg(d);
                                o = up ? 1.0 : 0.0;
                                di -= up ? 1 : -1;
                            }
                        }
                    }
                }
                v = nv;
                fm = __ldg(g.faces + v);
            }
        }
        const double rem = 1.0 - tau;
        o = dclamp01(o + times_nz<SANE>(rem, d));
        if (relax) A = A + times_any<SANE>(rem, rate);
        // ---- phase (Eq. 7)
        if (graded) {
            const double dx = times<SANE>((double)di + (o - o0), lp);
#pragma unroll
            for (int s = 0; s < NS; ++s)
                if (s < ctl.n_shapes)
                    ph[s] = ph[s] + times_any<SANE>(NS == 1 ? wg : __ldg(t.wG + (int64_t)s * t.n_steps + (k - 1)), dx);
        }
        // ---- displacement moments: the first warp sums the block's 32 walkers as
        //      the one-thread kernel's warp does
        if (k == next_rec) {
            s_mom[threadIdx.x >> 2][ax] = ax < 3 ? lp * ((double)di + (o - o0)) : A;
            __syncthreads();
            if (threadIdx.x < 32) {
                const double dx[3] = {s_mom[threadIdx.x][0], s_mom[threadIdx.x][1], s_mom[threadIdx.x][2]};
                const double Aw = s_mom[threadIdx.x][3];
                double al = Aw != 0.0 ? exp(-Aw) : 1.0;
                if ((int64_t)blockIdx.x * kQuadWalkers + threadIdx.x >= ctl.n_walkers) al = 0.0;
                warp_moments(al, dx, s_red);
                __syncwarp();
                if (threadIdx.x < kMoments)
                    ctl.mom_partial[((int64_t)rec * ctl.n_blocks * kWalkWarps + blockIdx.x) * kMoments + threadIdx.x] =
                        s_red[threadIdx.x];
            }
            __syncthreads();
            ++rec;
            next_rec = rec < ctl.n_rec ? __ldg(t.rec_step + rec) : INT32_MAX;
        }
    }

    if (active && ax < 3) {
        of_axis(st.o[0], st.o[1], st.o[2])[li] = o;
        of_axis(st.di[0], st.di[1], st.di[2])[li] = di;
#pragma unroll
        for (int s = 0; s < NS; ++s)
            if (s < ctl.n_shapes) st.phase[((int64_t)s * 3 + a) * ctl.n_walkers + li] = ph[s];
        if (ax == 0) {
            st.c[li] = c;
            st.A[li] = A;
        }
    }
}

}  // namespace rms
