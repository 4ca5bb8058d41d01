// btrt_tbn.cuh -- many time steps per launch for small lattices.
//
// On a lattice of some ten thousand nodes a step is about a microsecond of work for
// a fraction of the chip, while a launch costs 4 to 12 us whatever it computes (its
// code is fetched anew, its loads start cold).  Here one cooperative launch runs up
// to kTbnMaxSteps steps in rounds of `depth`: a block copies its output tile, grown by
// `depth` nodes on every side, from global to shared memory, advances the region
// `depth` steps there, one node less on every side with each, and writes the tile to
// the other buffer; a grid barrier ends the round.  The ring around a tile is
// recomputed by its neighbours: that costs arithmetic the idle chip has and buys one
// exchange per round instead of one per step.  Per node and step the arithmetic, and
// its order, is that of the one-step sweep and shared memory holds the stored form's
// values, so the results equal those of one step per launch bitwise.
//
// W threads cover a row of the region, so rows need no division: W = 32 for FP32
// compute (24 x 8 tiles at depth 4), 16 for FP64 and double-word (8 x 8 tiles), whose
// collisions are several hundred instructions and need spreading over more SMs.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "btrt_sweep.cuh"

namespace btrt {

constexpr int kTbnDepth = 4;         // most steps of one round
constexpr int kTbnMaxSteps = 256;    // most steps of one launch
constexpr int kTbnMaxThreads = 512;

// What differs between the steps of a launch, and its round structure.
template <typename Real>
struct TbnSteps {
    Real src_val[kTbnMaxSteps], wall_fac[kTbnMaxSteps];
    long long step0;            // step index that the first step produces
    int n, depth;               // steps of this launch, and of a round
    int ntx, ntiles;
    unsigned int *barrier;      // arrivals, zero at launch
    unsigned long long wait_limit;
};

template <typename Real, int SH> struct TbnGeom {
    static constexpr int W = sizeof(Real) == 4 ? 32 : 16;   // region width
    static constexpr int TY = 8;                            // output rows
    static constexpr int RH = TY + 2 * kTbnDepth;           // most region rows
    static constexpr int PLANE = RH * W;
    // nine populations, phi, and the form's own planes: the low words of phi, or the
    // writers' first moments
    static constexpr bool DW = PullShift<SH>::value == kShiftLocalDW, MOMENT = PullShift<SH>::value == kShiftMomentSR;
    static constexpr int VALS = 10 + (DW ? 1 : MOMENT ? 2 : 0);
    static constexpr int SMEM = 2 * VALS * PLANE * (int)sizeof(Real);
    static_assert(SMEM <= 48 * 1024, "fits the default per-block limit");
};

// A load that sees what other SMs wrote in earlier rounds (L1 is not coherent).
template <typename T> __device__ __forceinline__ T tbn_load(const T *ptr) {
    T v;
    if constexpr (sizeof(T) == 8) {
        const unsigned long long u = __ldcg(reinterpret_cast<const unsigned long long *>(ptr));
        memcpy(&v, &u, 8);
    } else if constexpr (sizeof(T) == 4) {
        const unsigned int u = __ldcg(reinterpret_cast<const unsigned int *>(ptr));
        memcpy(&v, &u, 4);
    } else {
        const unsigned short u = __ldcg(reinterpret_cast<const unsigned short *>(ptr));
        memcpy(&v, &u, 2);
    }
    return v;
}

// A region coordinate in the domain: wrapped on a periodic axis (once: both sides of
// the lattice are at least W), false beyond a wall, or `reach` nodes or more past the
// far side (nothing the tile still needs, and its neighbours were not computed).
__device__ __forceinline__ bool tbn_coord(int &g, int n, int wall, int reach) {
    if (g >= 0 && g < n) return true;
    if (wall || g >= n + reach) return false;
    g = g < 0 ? g + n : g - n;
    return true;
}

// Grid barrier of the round that brings the arrivals to `target`; all blocks are
// resident (cooperative launch).  Bounded wait: false, with flag bit 2 raised, when
// it gave up.
__device__ __forceinline__ bool tbn_barrier(unsigned int *count, unsigned int target, unsigned long long limit,
                                            int *flags) {
    __syncthreads();
    int good = 1;
    if (threadIdx.x == 0) {
        // releases the block's writes (ordered before by the barrier above); the acquiring
        // load and the barrier below order every thread's later loads
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        unsigned long long polls = 0;
        unsigned int seen;
        do {
            asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(seen) : "l"(count) : "memory");
            if (seen < target && ++polls > limit) {
                atomicOr(flags, 4);
                good = 0;
                break;
            }
        } while (seen < target);
    }
    return __syncthreads_and(good) != 0;
}

// Pull of a node from a shared-memory region (pull_node and pull_boundary on the
// region's values): the neighbours' values, then links that cross a bounce-back wall
// take the node's own opposite population and the wall term.
template <typename Real, int SH>
__device__ __forceinline__ void tbn_pull(const SweepParams<Real> &p, Real wall_fac, const Real *reg, int at, int gx, int gy,
                                         Real phi_prev, Real phi_lo, Real (&d)[9]) {
    using G = TbnGeom<Real, SH>;
    constexpr int PS = PullShift<SH>::value, PL = G::PLANE;
    constexpr bool LOCAL = PS == kShiftLocal || PS == kShiftLocalDW || PS == kShiftMomentSR;
    const Real *phr = reg + 9 * PL, *ext = reg + 10 * PL;   // phi; its low words, or the first moments
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const int nb = at - ey_of(i) * G::W - ex_of(i);
        d[i] = reg[BTRT_IX(p.flags, i * PL + nb, 9 * PL)];
        if (i == 0) continue;
        if constexpr (PS == kShiftLocal || PS == kShiftMomentSR) d[i] = fma(wgt<Real>(i), phr[nb] - phi_prev, d[i]);
        if constexpr (PS == kShiftMomentSR) d[i] = fma(w3<Real>(i), e_dot<Real>(i, ext[nb], ext[PL + nb]), d[i]);
        if constexpr (PS == kShiftLocalDW)
            d[i] = fma(wgt<Real>(i), (phr[nb] - phi_prev) + (ext[nb] - phi_lo), d[i]);
    }
    const bool x0 = p.hbb_x && gx == 0, x1 = p.hbb_x && gx == p.nx - 1;
    const bool y0 = p.hbb_y && gy == 0, y1 = p.hbb_y && gy == p.ny - 1;
    if (!(x0 || x1 || y0 || y1)) return;
    auto value = [&](int side, int idx) {
        const Real *a = p.wall_arr[side];
        return (a ? a[BTRT_IX(p.flags, idx, side < 2 ? p.ny : p.nx)] : p.wall_const[side]) * wall_fac;
    };
    Real vx = Real(0), vy = Real(0);
    if (x0 || x1) vx = value(x0 ? 0 : 1, gy);
    if (y0 || y1) vy = value(y0 ? 2 : 3, gx);
#pragma unroll
    for (int i = 1; i < 9; ++i) {
        const bool cx = (ex_of(i) == 1 && x0) || (ex_of(i) == -1 && x1);
        const bool cy = (ey_of(i) == 1 && y0) || (ey_of(i) == -1 && y1);
        if (!cx && !cy) continue;
        const Real phi_w = cx && cy ? Real(0.5) * (vx + vy) : (cy ? vy : vx);
        const Real dout = reg[BTRT_IX(p.flags, opp_of(i) * PL + at, 9 * PL)];
        Real wt = wall_term(p, opp_of(i), phi_w);
        if constexpr (PS == kShiftRef) wt = wt - Real(2) * p.wref[i];
        if constexpr (LOCAL) wt = fma(Real(-2) * wgt<Real>(i), phi_prev, wt);
        if constexpr (PS == kShiftLocalDW) wt = fma(Real(-2) * wgt<Real>(i), phi_lo, wt);
        d[i] = wt - dout;
        if constexpr (PS == kShiftMomentSR) d[i] = fma(w3<Real>(i), e_dot<Real>(i, ext[at], ext[PL + at]), d[i]);
    }
}

// Threads and resident blocks per SM the kernel is compiled for.  FP32 compute: two
// blocks of 512 (64 registers), so that four of 256 fit as well: us per step at 256^2,
// FP32 storage, manufactured solution / nonlinear 2.45 / 2.35 against 4.03 / 3.97 with the
// compiler's 80 registers (64^2: 1.59 / 1.45 against 1.54 / 1.42).  Double-word, constant
// coefficients: three of 256, 181^2 3.1 against 4.3 with two; its per-node coefficients
// (160^2 3.5 against 4.6 with three) and FP64 (64^2 hill 2.0 against 2.1) two.
template <typename Real, int MODE> struct TbnBounds {
    static constexpr int threads = sizeof(Real) == 4 ? kTbnMaxThreads : 256;
    static constexpr int blocks = std::is_same<Real, dw>::value && MODE != kGeneral ? 3 : 2;
};

// st.n steps: p holds the parameters of the first (its inputs in fin, phi_in; the
// other buffers in fout, phi_out; the rounds swap them).
template <typename Real, typename S, int SH, int MODE, int SRC>
__global__ void __launch_bounds__(TbnBounds<Real, MODE>::threads, TbnBounds<Real, MODE>::blocks)
    sweep_tbn_kernel(const __grid_constant__ SweepParams<Real> p, const __grid_constant__ TbnSteps<Real> st) {
    using G = TbnGeom<Real, SH>;
    constexpr int SC = CollShift<SH>::value, PL = G::PLANE;
    const int step_rows = blockDim.x / G::W;          // region rows covered at a time
    extern __shared__ __align__(16) unsigned char tbn_smem[];
    Real *buf = reinterpret_cast<Real *>(tbn_smem);   // [2][VALS][RH][W]
    const int lx = threadIdx.x % G::W, row0 = threadIdx.x / G::W;
    const int tx = G::W - 2 * st.depth;
    bool bad = false;
    unsigned int target = 0;
    for (int k = 0; k < st.n; k += st.depth) {
        const int r = min(st.depth, st.n - k);        // steps of this round
        const bool odd = (k / st.depth) & 1;
        const S *fin = static_cast<const S *>(odd ? p.fout : p.fin);
        S *fout = odd ? static_cast<S *>(const_cast<void *>(p.fin)) : static_cast<S *>(p.fout);
        const Real *phi_in = odd ? p.phi_out : p.phi_in;
        Real *phi_out = odd ? const_cast<Real *>(p.phi_in) : p.phi_out;
        for (int tile = blockIdx.x; tile < st.ntiles; tile += gridDim.x) {
            const int x0 = (tile % st.ntx) * tx - r, y0 = (tile / st.ntx) * G::TY - r;
            const int width = tx + 2 * r, rows = G::TY + 2 * r;
            int gx = x0 + lx;
            const bool in_x = lx < width && tbn_coord(gx, p.nx, p.hbb_x, r);
            Real xs = Real(0), xc = Real(0);
            if (in_x && SRC != kSrcReaction && p.src_kind == kSrcTrig) {
                xs = p.Xs[BTRT_IX(p.flags, gx, p.nx)];
                xc = p.Xc[BTRT_IX(p.flags, gx, p.nx)];
            }
            // the region's stored values and phi
            if (in_x)
                for (int ly = row0; ly < rows; ly += step_rows) {
                    int gy = y0 + ly;
                    if (!tbn_coord(gy, p.ny, p.hbb_y, r)) continue;
                    const int node = gy * p.pitch + gx, at = ly * G::W + lx;
                    S v[9];
#pragma unroll
                    for (int i = 0; i < 9; ++i) v[i] = tbn_load(fin + BTRT_IX(p.flags, i * p.plane + node, 9 * p.plane));
                    buf[9 * PL + at] = tbn_load(phi_in + BTRT_IX(p.flags, node, p.plane));
                    if constexpr (G::DW)
                        buf[10 * PL + at] = tbn_load((odd ? p.phi_out_lo : p.phi_in_lo) + BTRT_IX(p.flags, node, p.plane));
                    if constexpr (G::MOMENT) {
                        const S *j = static_cast<const S *>(odd ? p.j_out : p.j_in);
                        buf[10 * PL + at] = dev_load<Real, S, SH>(tbn_load(j + BTRT_IX(p.flags, node, 2 * p.plane)));
                        buf[11 * PL + at] = dev_load<Real, S, SH>(tbn_load(j + BTRT_IX(p.flags, p.plane + node, 2 * p.plane)));
                    }
#pragma unroll
                    for (int i = 0; i < 9; ++i) buf[i * PL + at] = dev_load<Real, S, SH>(v[i]);
                }
            __syncthreads();
            for (int s = 1; s <= r; ++s) {
                const bool last = s == r;
                const Real *in = buf + (s & 1 ? 0 : G::VALS * PL);
                Real *out = buf + (s & 1 ? G::VALS * PL : 0);
                const Real src_val = st.src_val[k + s - 1], wall_fac = st.wall_fac[k + s - 1];
                if (in_x && lx >= s && lx < width - s && x0 + lx < p.nx + r - s) {
#pragma unroll 1
                    for (int ly = s + row0; ly < rows - s; ly += step_rows) {
                        int gy = y0 + ly;
                        if (!tbn_coord(gy, p.ny, p.hbb_y, r - s)) continue;
                        const int node = gy * p.pitch + gx, at = ly * G::W + lx;
                        Real d[9];
                        const Real phi_prev = in[9 * PL + at];
                        Real phi_lo = Real(0);
                        if constexpr (G::DW) phi_lo = in[10 * PL + at];
                        tbn_pull<Real, SH>(p, wall_fac, in, at, gx, gy, phi_prev, phi_lo, d);
                        const Real srcv = source_at<Real, SRC>(p, xs, xc, gy, node);
                        const Real rs = SC == kShiftLocal ? phi_prev : p.phi_ref;
                        Real phid, phi;
                        if constexpr (std::is_same<Real, double>::value) {
                            phi = collide_f64<MODE, SRC, true>(p, d, phi_prev, srcv, node, src_val);
                            phid = phi;
                        } else {
                            phi = collide_fold<Real, MODE, SRC, SC>(p, d, rs, phi_prev, srcv, false, node, phid, nullptr,
                                                                    &src_val);
                        }
                        // the stored form, as finish_node forms it
                        S v[9];
                        unsigned int h = 0;
                        if constexpr (StoreSR<SH>::value) h = sr_node_bits(sr_step_seed(st.step0 + k + s - 1), node);
                        S jx, jy;
                        if constexpr (G::MOMENT) {
                            jx = j_pack<S, SH>(((d[1] - d[3]) + (d[5] - d[7])) + (d[8] - d[6]));
                            jy = j_pack<S, SH>(((d[2] - d[4]) + (d[5] - d[7])) + (d[6] - d[8]));
                            const Real jxv = dev_load<Real, S, SH>(jx), jyv = dev_load<Real, S, SH>(jy);
#pragma unroll
                            for (int i = 0; i < 9; ++i) {
                                Real t = fma(-wgt<Real>(i), phid, d[i]);
                                if (i != 0) t = fma(-w3<Real>(i), e_dot<Real>(i, jxv, jyv), t);
                                v[i] = pack_sr_sub<S>(t, sr_bits(h, i));
                            }
                            phi = phi_sr(phi, phid, rs, sr_bits(h, 9));
                        } else if constexpr (StoreSR<SH>::value) {
#pragma unroll
                            for (int i = 0; i < 9; ++i) v[i] = pack_sr<S>(fma(-wgt<Real>(i), phid, d[i]), sr_bits(h, i));
                        } else {
#pragma unroll
                            for (int i = 0; i < 9; ++i) v[i] = store_value<Real, S, SC>(i, d[i], phid);
                        }
                        Real lo = Real(0);
                        if constexpr (G::DW) {
                            const Real bb = phi - phi_prev;
                            const Real e = (phi_prev - (phi - bb)) + (phid - bb);
                            const Real l = phi_lo + e;
                            const Real hi = phi + l;
                            lo = l - (hi - phi);
                            phi = hi;
                        }
                        bad |= not_finite(phi);
                        if (last) {
#pragma unroll
                            for (int i = 0; i < 9; ++i) fout[BTRT_IX(p.flags, i * p.plane + node, 9 * p.plane)] = v[i];
                            phi_out[BTRT_IX(p.flags, node, p.plane)] = phi;
                            if constexpr (G::DW)
                                (odd ? const_cast<Real *>(p.phi_in_lo) : p.phi_out_lo)[BTRT_IX(p.flags, node, p.plane)] = lo;
                            if constexpr (G::MOMENT) {
                                S *j = static_cast<S *>(odd ? const_cast<void *>(p.j_in) : p.j_out);
                                j[BTRT_IX(p.flags, node, 2 * p.plane)] = jx;
                                j[BTRT_IX(p.flags, p.plane + node, 2 * p.plane)] = jy;
                            }
                        } else {
#pragma unroll
                            for (int i = 0; i < 9; ++i) out[i * PL + at] = dev_load<Real, S, SH>(v[i]);
                            out[9 * PL + at] = phi;
                            if constexpr (G::DW) out[10 * PL + at] = lo;
                            if constexpr (G::MOMENT) {
                                out[10 * PL + at] = dev_load<Real, S, SH>(jx);
                                out[11 * PL + at] = dev_load<Real, S, SH>(jy);
                            }
                        }
                    }
                }
                __syncthreads();
            }
        }
        if (k + st.depth < st.n) {
            target += gridDim.x;
            if (!tbn_barrier(st.barrier, target, st.wait_limit, p.flags)) break;
        }
    }
    if (bad) atomicOr(p.flags, 1);
}

// Resident blocks of an instantiation with `threads` threads (256 or 512), measured
// once per device; negative: an error.
template <typename Real, typename S, int SH, int MODE, int SRC>
int tbn_resident(int threads, cudaError_t &e) {
    constexpr int kMaxDev = 64;
    static std::mutex mu;
    static int of[kMaxDev][2] = {};
    int dev = 0;
    e = cudaGetDevice(&dev);
    if (e == cudaSuccess && (dev < 0 || dev >= kMaxDev)) e = cudaErrorInvalidDevice;
    if (e != cudaSuccess) return -1;
    std::lock_guard<std::mutex> lock(mu);
    int &n = of[dev][threads == kTbnMaxThreads];
    if (!n) {
        int per_sm = 0, sms = 0;
        e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sweep_tbn_kernel<Real, S, SH, MODE, SRC>, threads,
                                                              TbnGeom<Real, SH>::SMEM);
        if (e == cudaSuccess && per_sm < 1) e = cudaErrorInvalidConfiguration;
        if (e != cudaSuccess) return -1;
        n = per_sm * sms;
    }
    return n;
}

template <typename Real, typename S, int SH, int MODE, int SRC>
cudaError_t launch_tbn_src(const SweepParams<Real> &p, TbnSteps<Real> &st, int *rounds, cudaStream_t s) {
    using G = TbnGeom<Real, SH>;
    // The deepest rounds whose tiles are all resident at once (a second wave of tiles
    // costs more than the deeper round saves); FP32 compute takes 512 threads, one
    // region row per warp, where those still fit at full depth.
    const int deepest = std::min(st.n, kTbnDepth);
    int threads = 256, blocks = 0;
    cudaError_t e = cudaSuccess;
    auto tiles = [&](int depth) {
        const int tx = G::W - 2 * depth;
        st.depth = depth;
        st.ntx = (p.nx + tx - 1) / tx;
        st.ntiles = st.ntx * ((p.ny + G::TY - 1) / G::TY);
        return st.ntiles;
    };
    if (G::W == 32) {
        blocks = tbn_resident<Real, S, SH, MODE, SRC>(kTbnMaxThreads, e);
        if (e != cudaSuccess) return e;
        if (tiles(deepest) <= blocks) threads = kTbnMaxThreads;
    }
    if (threads == 256) {
        blocks = tbn_resident<Real, S, SH, MODE, SRC>(256, e);
        if (e != cudaSuccess) return e;
        for (int depth = deepest; tiles(depth) > blocks && depth > 2; --depth) {}
    }
    *rounds = (st.n + st.depth - 1) / st.depth;
    auto *kernel = sweep_tbn_kernel<Real, S, SH, MODE, SRC>;
    const dim3 grid((unsigned)std::min(st.ntiles, blocks)), block((unsigned)threads);
    if (*rounds == 1) {   // no block waits
        kernel<<<grid, block, G::SMEM, s>>>(p, st);
        return cudaGetLastError();
    }
    e = cudaMemsetAsync(st.barrier, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) return e;
    void *args[] = {const_cast<SweepParams<Real> *>(&p), &st};
    return cudaLaunchCooperativeKernel(reinterpret_cast<const void *>(kernel), grid, block, args, G::SMEM, s);
}

template <typename Real, typename S, int SH>
cudaError_t launch_tbn_sh(const SweepParams<Real> &p, TbnSteps<Real> &st, int mode, int *rounds, cudaStream_t s) {
    const bool react = p.src_kind == kSrcReaction;
    if (mode == kGeneral)
        return react ? launch_tbn_src<Real, S, SH, kGeneral, kSrcReaction>(p, st, rounds, s)
                     : launch_tbn_src<Real, S, SH, kGeneral, kSrcRuntimeNR>(p, st, rounds, s);
    return react ? launch_tbn_src<Real, S, SH, kLinear, kSrcReaction>(p, st, rounds, s)
                 : launch_tbn_src<Real, S, SH, kLinear, kSrcRuntimeNR>(p, st, rounds, s);
}

// FP32 compute with storage S, every stored form it has.
template <typename S>
cudaError_t launch_tbn_storage(const SweepParams<float> &p, TbnSteps<float> &st, int shift, int mode, int *rounds,
                               cudaStream_t s) {
    switch (shift) {
    case kShiftRef: return launch_tbn_sh<float, S, kShiftRef>(p, st, mode, rounds, s);
    case kShiftLocal: return launch_tbn_sh<float, S, kShiftLocal>(p, st, mode, rounds, s);
    case kShiftLocalDW: return launch_tbn_sh<float, S, kShiftLocalDW>(p, st, mode, rounds, s);
    }
    if constexpr (!std::is_same<S, float>::value) {
        if (shift == kShiftLocalSR) return launch_tbn_sh<float, S, kShiftLocalSR>(p, st, mode, rounds, s);
        if (shift == kShiftLocalDWSR) return launch_tbn_sh<float, S, kShiftLocalDWSR>(p, st, mode, rounds, s);
        if (shift == kShiftMomentSR) return launch_tbn_sh<float, S, kShiftMomentSR>(p, st, mode, rounds, s);
    }
    return cudaErrorInvalidValue;
}

}  // namespace btrt
