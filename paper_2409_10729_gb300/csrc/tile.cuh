// tile.cuh -- the sweep of one direction as a sequence of block-wide passes
// over a tile of cells held in shared memory.
//
// A tile is P adjacent pencils (P a power of two) by J cells along the sweep
// direction.  The block
//   A  loads the tile's cells and three more on either side, converts them to
//      primitives and stores those,
//   B  reconstructs both face values of the J + 2 cells -1 .. J, one field of
//      a short run of double cells per thread at a time (what neighbouring cells
//      share is carried along the run),
//   C  solves HLLC at the J + 1 faces, one face per thread,
//   D  forms L for the J cells and finishes them (accumulator, stage update,
//      wave speed).
// The FP64 form is bound by the FP64 pipe (2 lanes per SM and clock) as long as
// enough warps are in flight.  A thread that slides a five-cell window of all
// fields along its pencil needs 255 registers, 8 warps per SM, and reached 55
// to 60% of that pipe once the quotients had moved to the integer pipes; one
// field at a time from shared memory needs 100, 16 warps, and reaches 80 to 84%
// (128^3, ncu: 547 FP64 of 9975 instructions per 32 cells and 0.96 issued per
// clock with WENO's and HLLC's quotients on the integer pipes; 440 and 1.7 with
// WENO's products and HLLC's square roots there too).  It also gives small grids
// parallel work: a thread's serial chain is R reconstructions and one flux
// instead of a segment of whole cells, and a single pencil fills its warps with
// cells along it.  Measured, sliding window
// -> tiles: 256^3 droplets 0.557 -> 0.464 ns per cell, equation and RHS;
// 1024x512 column 6.72 -> 3.36 ms a step; 32^3 RHS 3.9 -> 0.18 ms; 1000-cell
// tube 2.67 -> 0.041 ms a step.  (256^3 0.39 now, with WENO's products off the
// FP64 pipe too, physics_exact.cuh, and the shapes of pick_tile.)
#pragma once
#include <algorithm>
#include <atomic>

#include "sweep.cuh"

namespace mfc5 {

constexpr int kTileThreads = 128;

// Tiles resident per SM: the register allocator's cap (128 registers a thread;
// the kernels use 96 to 128, without spills) and the share of an SM's shared
// memory (228 KB, 1 KB of it reserved per block) that a tile may take.
#ifndef MFC_TILE_BLOCKS
#define MFC_TILE_BLOCKS 4
#endif
constexpr int kTileSmem = 228 * 1024;

struct TileShape {
    int lp;          // log2 P
    int J, R;
    int ntp;         // tiles across the pencils
    long long npen;  // pencils
};

// Values of shared memory of a tile.
__host__ __device__ inline size_t tile_elems(int neq, int P, int J) {
    const int ps = P > 1 ? P + 1 : 1;   // odd pitch: no bank conflicts along either index
    return (size_t)neq * ps * ((J + 6) + 2 * (J + 2));
}

// Finishes cell c (index j along the sweep direction) with L = L_DIR(q) of
// this sweep: accumulate, or the SSP-RK3 stage update and, on stage 3, the
// cell's wave speed.
template <int NDIM, int DIR, int MODE, bool NU, int NF>
__device__ __forceinline__ void finish_cell(const SweepArgs& a, double dt, const double* L, long long c, int j,
                                              long long pencil, double& smax, bool& bad) {
    using FL = Fields<NDIM, NF>;
    constexpr int NEQ = FL::NEQ;
    const long long nc = a.ncell;
    double* acc = static_cast<double*>(a.acc);
    if constexpr (MODE == SW_FIRST) {
#pragma unroll
        for (int f = 0; f < NEQ; ++f) acc[f * nc + c] = L[f];
    } else if constexpr (MODE == SW_MID) {
#pragma unroll
        for (int f = 0; f < NEQ; ++f) acc[f * nc + c] = acc[f * nc + c] + L[f];
    } else if constexpr (MODE == SW_LAST_RHS) {
        double* out = static_cast<double*>(a.qout);
#pragma unroll
        for (int f = 0; f < NEQ; ++f) out[f * nc + c] = NDIM > 1 ? acc[f * nc + c] + L[f] : L[f];
    } else {
        const double* qin = static_cast<const double*>(a.qin);
        double* out = static_cast<double*>(a.qout);
        double qnew[NEQ];
#pragma unroll
        for (int f = 0; f < NEQ; ++f) {
            const double tot = NDIM > 1 ? acc[f * nc + c] + L[f] : L[f];
            const double qn = a.qn[f * nc + c];
            const double dL = dt * tot;
            if (a.stage == 1) {
                qnew[f] = qn + dL;
            } else {
                const double qk = qin[f * nc + c];
                if (a.stage == 2) qnew[f] = 0.75 * qn + 0.25 * (qk + dL);
                else qnew[f] = (1.0 / 3.0) * qn + (2.0 / 3.0) * (qk + dL);
            }
        }
#pragma unroll
        for (int f = 0; f < NEQ; ++f) out[f * nc + c] = qnew[f];
        if (a.stage == 3) {
            double s, dx3[3], rdx3[3], idx3[3];
            // the pencil's position in the plane normal to DIR, x (or y) fastest
            int ia = 0, b = 0;
            if (NU) {
                const int na = DIR == 0 ? a.n[1] : a.n[0];
                ia = (int)(pencil % na);
                b = (int)(pencil / na);
            }
            cell_geometry<DIR, NU>(a, j, ia, b, dx3, rdx3, idx3);
            s = exact::cell_wavespeed<NDIM, NF>(a.eos, qnew, dx3, rdx3, bad);
            smax = s > smax ? s : smax;
        }
    }
}

template <int NDIM, int DIR, int MODE, bool NU, int NF>
__global__ void __launch_bounds__(kTileThreads, MFC_TILE_BLOCKS) tile_kernel(const SweepArgs a, const TileShape ts) {
    constexpr int T = kTileThreads;
    using FL = Fields<NDIM, NF>;
    constexpr int NEQ = FL::NEQ, IA = FL::IA, NA = FL::NA;
    extern __shared__ double tsm[];
    const int P = 1 << ts.lp, PS = P > 1 ? P + 1 : 1;
    const int ns = a.n[DIR];
    const long long nc = a.ncell;
    const long long ss = DIR == 0 ? 1LL : (DIR == 1 ? (long long)a.n[0] : (long long)a.n[0] * a.n[1]);
    const int tj = (int)(blockIdx.x / ts.ntp);
    const long long pen0 = (long long)(blockIdx.x - (unsigned)tj * ts.ntp) << ts.lp;
    const int j0 = tj * ts.J;
    const int Jc = min(ts.J, ns - j0);
    const int wf = (ts.J + 6) * PS, vf = (ts.J + 2) * PS;   // field pitches
    double* const W = tsm;
    double* const VM = W + NEQ * wf;   // value at i+1/2 of cell row r (cell j0 - 1 + r)
    double* const VP = VM + NEQ * vf;  // value at i-1/2; then the flux through that face
    bool bad = false;
    double smax = 0.0;

    // first cell of pencil id (its position in the plane normal to DIR)
    auto pencil_base = [&](long long id) -> long long {
        if constexpr (DIR == 0) return id * a.n[0];
        else if constexpr (DIR == 1) {
            const long long row = ts.npen < (1LL << 32) ? (long long)((unsigned)id / (unsigned)a.n[0]) : id / a.n[0];
            return id - row * a.n[0] + row * ((long long)a.n[0] * a.n[1]);
        }
        else return id;
    };

    // A: primitives of cells j0 - 3 .. j0 + Jc + 2 (ghosts from the neighbour
    // block's halo, or from the BC index map)
    {
        const int rows = Jc + 6;
        for (int it = threadIdx.x; it < rows << ts.lp; it += T) {
            const int p = DIR == 0 ? it / rows : it & (P - 1), r = DIR == 0 ? it - p * rows : it >> ts.lp;
            const bool active = pen0 + p < ts.npen;
            const long long id = active ? pen0 + p : ts.npen - 1;
            const int j = j0 - 3 + r;
            const double* src = static_cast<const double*>(a.qin);
            long long c, fs = nc;
            const double* h = j < 0 ? static_cast<const double*>(a.hlo) : (j >= ns ? static_cast<const double*>(a.hhi) : nullptr);
            if (h) {
                src = h;
                c = (long long)(j < 0 ? j + 3 : j - ns) * a.hplane + id;
                fs = 3 * a.hplane;
            } else {
                c = pencil_base(id) + (long long)bc_index(j, ns, a.periodic) * ss;
            }
            double v[NEQ], w[NEQ];
#pragma unroll
            for (int f = 0; f < NEQ; ++f) v[f] = __ldg(src + f * fs + c);
            exact::cons_to_prim<NDIM, NF>(a.eos, v, w);
            bad |= active && !pos(mix_rho<NF>(w));
#pragma unroll
            for (int f = 0; f < NEQ; ++f) W[f * wf + r * PS + p] = w[f];
        }
    }
    __syncthreads();
    // B: reconstruction, one field of a run of double cells per thread
    {
        const int rows = Jc + 2, nrun = (rows + ts.R - 1) / ts.R;
        for (int it = threadIdx.x; it < (NEQ * nrun) << ts.lp; it += T) {
            const int p = it & (P - 1), q = it >> ts.lp, f = q / nrun, r0 = (q - f * nrun) * ts.R;
            const int r1 = min(r0 + ts.R, rows);
            const double* w = W + f * wf + r0 * PS + p;
            double* vm = VM + f * vf + r0 * PS + p;
            double* vp = VP + f * vf + r0 * PS + p;
            double v0 = w[0], v1 = w[PS], v2 = w[2 * PS], v3 = w[3 * PS];
            w += 4 * PS;
            const bool nu = NU && a.tab, w5 = a.order == 5;
            // carried along the run: curvature terms and right-face candidates
            double t0 = 0.0, t1 = 0.0, p0 = 0.0, p1 = 0.0;
            if (!nu && w5) {
                t0 = exact::curv(v0, v1, v2);
                t1 = exact::curv(v1, v2, v3);
                exact::weno5_right01(v0, v1, v2, v3, p0, p1);
            }
#pragma unroll 1
            for (int r = r0; r < r1; ++r) {
                const double v4 = *w;
                double m, q5;
                if (nu) {
                    const double* T5 = static_cast<const double*>(a.tab) + (long long)(j0 + r) * kTabDoubles;
                    exact::weno5_tab(T5, v0, v1, v2, v3, v4, a.eps, m, q5);
                } else if (w5) {
                    const double t2 = exact::curv(v2, v3, v4);
                    exact::weno5_tc(a.eps, v0, v1, v2, v3, v4, t0, t1, t2, p0, p1, m, q5);
                    t0 = t1;
                    t1 = t2;
                } else {
                    exact::weno3(a.eps, v1, v2, v3, m, q5);
                }
                *vm = m;
                *vp = q5;
                v0 = v1;
                v1 = v2;
                v2 = v3;
                v3 = v4;
                w += PS;
                vm += PS;
                vp += PS;
            }
        }
    }
    __syncthreads();
    // C: the flux through face j (between cell rows j and j + 1) replaces the
    // right state it was formed from; the region velocity goes to VM[0] row j
    for (int it = threadIdx.x; it < (Jc + 1) << ts.lp; it += T) {
        double F[NEQ], uf;
        const int o = (it >> ts.lp) * PS + (it & (P - 1));
        const bool fb = exact::hllc<NDIM, DIR, NF>(a.eos, VM + o, VP + o + PS, vf, F, uf);
        bad |= fb && pen0 + (it & (P - 1)) < ts.npen;
#pragma unroll
        for (int f = 0; f < NEQ; ++f) VP[f * vf + o + PS] = F[f];
        VM[o] = uf;
    }
    __syncthreads();
    // D: divergence of the cells (row j + 1: face j below, face j + 1 above)
    {
        const double dt = MODE == SW_LAST_RK ? a.ctrl->dt : 0.0;
        const unsigned dxh = (unsigned)__double2hiint(a.dx[DIR]), dxe = (dxh >> 20) & 0x7ffu;
        const bool pow2_dx = (dxh & 0x800fffffu) == 0u && __double2loint(a.dx[DIR]) == 0 && dxe - 2u < 2043u;
        for (int it = threadIdx.x; it < Jc << ts.lp; it += T) {
            const int p = DIR == 0 ? it / Jc : it & (P - 1), r = DIR == 0 ? it - p * Jc : it >> ts.lp;
            const long long id = pen0 + p;
            if (id >= ts.npen) continue;
            const int o = r * PS + p, j = j0 + r;
            const double* F = VP + o + PS;
            const double du = VM[o + PS] - VM[o];
            double L[NEQ];
            double dx = a.dx[DIR], rdx = a.rdx[DIR];
            if (NU && a.cw[DIR]) {   // non-uniform: the cell's own width
                dx = __ldg(a.cw[DIR] + j);
                rdx = __ldg(a.crw[DIR] + j);
            }
            if (pow2_dx && !(NU && a.cw[DIR])) {
                // a power-of-two width: x / dx and x * (1/dx) are the same real
                // number, so one multiplication gives the quotient's bits
#pragma unroll
                for (int f = 0; f < NEQ; ++f) L[f] = (F[f * vf] - F[f * vf + PS]) * rdx;
#pragma unroll
                for (int i = 0; i < NA; ++i)
                    L[IA + i] = L[IA + i] + W[(IA + i) * wf + o + 3 * PS] * du * rdx;
            } else {
#pragma unroll
                for (int f = 0; f < NEQ; ++f) L[f] = exact::div_rcp(F[f * vf] - F[f * vf + PS], dx, rdx);
#pragma unroll
                for (int i = 0; i < NA; ++i)
                    L[IA + i] = L[IA + i] + exact::div_rcp(W[(IA + i) * wf + o + 3 * PS] * du, dx, rdx);
            }
            const long long c = pencil_base(id) + (long long)j * ss;
            finish_cell<NDIM, DIR, MODE, NU, NF>(a, dt, L, c, j, id, smax, bad);
        }
    }
    const int lane = threadIdx.x & 31;
    if constexpr (MODE == SW_LAST_RK) {
        if (a.stage == 3) {
            const double m = warp_max(smax);
            if (lane == 0 && m > 0.0)
                atomicMax(&a.ctrl->S_bits, (unsigned long long)__double_as_longlong(m));
        }
    }
    if (__any_sync(0xffffffffu, bad) && lane == 0) atomicOr(&a.ctrl->status, 1u);
}

// Tile of a launch.  Large grids: the split with the least FP64 work per cell, by
// counting.  A pass over w warps' worth of items costs its warps, and, because a
// block's four warps meet at a barrier after it, its rounds of four; the FP64
// instructions of one item are about 8 + 31 R for a run of R reconstructions, 114
// for a flux, 20 for a conversion and 25 for a cell's end.  P = 4 or 8, pencils
// cut evenly into up to four pieces more than shared memory asks for, R = 3..9;
// the estimate is the larger of the rounds and 1.1 times the warps (the FP64 pipe
// is busy 0.8 of the time at best).  Measured against P = 4, J <= 64, R = 4
// everywhere: 256^3 144.6 -> 140.0 ms a step, 203^3 80.1 -> 74.9, 160^3 39.3 ->
// 37.0, 131^3 25.3 -> 24.2, 96^3 10.8 -> 10.5, 1024x512 2.86 -> 2.70 (fixed splits
// ranged from 140 to 179 ms at 256^3).
// Grids with fewer than three tiles per resident block at P = 4: J is halved
// from 64 down to 16 cells (8 on a single pencil), so that small grids use the
// whole device, and the runs are shortened, which trades the terms that cells
// share for a shorter serial chain: 32^3 0.454 ms a step with P 4, J 16, R 2 (4,
// 32, 2: 0.525; 8, 16, 3: 0.545; 2, 16, 2: 0.479); 1000 cells in 1-D 0.041 ms a
// step for J 8 or 16 (32: 0.052).
inline TileShape pick_tile(int dir, const int* n, long long ncell, int neq, long long slots) {
    TileShape t;
    const int ns = n[dir];
    t.npen = ncell / ns;
    auto most_cells = [&](int lp) {   // J that shared memory allows
        const int ps = lp ? (1 << lp) + 1 : 1;
        return ((int)(kTileSmem / MFC_TILE_BLOCKS - 1024) / 8 / (neq * ps) - 10) / 3;
    };
    auto across = [&](int lp) { return (int)((t.npen + (1LL << lp) - 1) >> lp); };
    t.lp = t.npen >= 4 ? 2 : (t.npen >= 2 ? 1 : 0);
    t.ntp = across(t.lp);
    int most = std::min(most_cells(t.lp), 64);
    const int least = t.npen == 1 ? 8 : 16;
    auto tiles = [&](int J) { return (long long)t.ntp * ((ns + J - 1) / J); };
    if (tiles(most) < 3 * slots || t.lp < 2) {
        while (most / 2 >= least && tiles(most) < 3 * slots) most /= 2;
        const int nt = (ns + most - 1) / most;
        t.J = (ns + nt - 1) / nt;
        const long long nb = tiles(t.J);
        t.R = nb >= 3 * slots ? 4 : (2 * nb >= slots ? 2 : 1);
        return t;
    }
    double best = 0.0;
    int blp = 2, bJ = 0, bR = 4;
    for (int lp = 2; lp <= 3 && (1LL << lp) <= t.npen; ++lp) {
        const int P = 1 << lp, nt0 = (ns + most_cells(lp) - 1) / most_cells(lp);
        int last = 0;
        for (int nt = nt0; nt < nt0 + 5; ++nt) {
            const int J = (ns + nt - 1) / nt;
            if (nt > nt0 && (J < 8 || J == last)) break;
            last = J;
            for (int R = 3; R <= 9; ++R) {
                const int w[4] = {(neq * ((J + 2 + R - 1) / R) * P + 31) / 32, ((J + 1) * P + 31) / 32,
                                  ((J + 6) * P + 31) / 32, (J * P + 31) / 32};
                const int c[4] = {8 + 31 * R, 114, 20, 25};
                int pipe = 0, rounds = 0;
                for (int k = 0; k < 4; ++k) {
                    pipe += w[k] * c[k];
                    rounds += (w[k] + 3) / 4 * 4 * c[k];
                }
                const double cost = std::max(1.1 * pipe, (double)rounds) * across(lp) * ((ns + J - 1) / J);
                if (bJ == 0 || cost < best) {
                    best = cost;
                    blp = lp;
                    bJ = J;
                    bR = R;
                }
            }
        }
    }
    t.lp = blp;
    t.ntp = across(blp);
    t.J = bJ;
    t.R = bR;
    return t;
}

// Lets the kernel use the SM's shared memory (once per kernel and device) and
// returns the device's tile slots, MFC_TILE_BLOCKS per SM.
template <int NDIM, int DIR, int MODE, bool NU, int NF>
cudaError_t tile_slots(long long* slots) {
    constexpr int kMaxDev = 64;
    static std::atomic<int> sms_of[kMaxDev];   // 0: not yet set up
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    int sms = dev >= 0 && dev < kMaxDev ? sms_of[dev].load(std::memory_order_acquire) : 0;
    if (sms == 0) {
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(tile_kernel<NDIM, DIR, MODE, NU, NF>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, kTileSmem / MFC_TILE_BLOCKS);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < kMaxDev) sms_of[dev].store(sms, std::memory_order_release);
    }
    *slots = (long long)sms * MFC_TILE_BLOCKS;
    return cudaSuccess;
}

template <int NDIM, int DIR, int MODE, bool NU, int NF>
cudaError_t launch_tile(const SweepArgs& a, cudaStream_t s) {
    constexpr int NEQ = Fields<NDIM, NF>::NEQ;
    long long slots = 0;
    cudaError_t e = tile_slots<NDIM, DIR, MODE, NU, NF>(&slots);
    if (e != cudaSuccess) return e;
    const TileShape t = pick_tile(DIR, a.n, a.ncell, NEQ, slots);
    const size_t smem = tile_elems(NEQ, 1 << t.lp, t.J) * sizeof(double);
    if (a.dry) return cudaSuccess;
    const long long blocks = (long long)t.ntp * ((a.n[DIR] + t.J - 1) / t.J);
    if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
    tile_kernel<NDIM, DIR, MODE, NU, NF><<<(unsigned)blocks, kTileThreads, smem, s>>>(a, t);
    return cudaGetLastError();
}

}  // namespace mfc5
