// rk4ip_2d_tma.cu -- the complex64 2D passes as persistent, TMA-pipelined kernels.
//
// Same arithmetic as rk4ip_2d.cu (XMDS2 Sec. 2.6: exp(L dt/2) in Fourier space,
// the real-space RK4 stages in between; Sec. 2.2: separable transforms), laid
// out for sm_103a: persistent CTAs walk a list of work items; shared-memory stages
// hold the item being transformed and the next ones, which the
// tensor-memory-access unit is already copying in (cp.async.bulk, completion
// on an mbarrier with a byte count), so that no register holds data in flight.
//   row item    : ROWS lines of A and of B (1D bulk copies, 2 x 8 KB, four CTAs an SM);
//                 each FFT runs in place in the staged lines, the result leaves
//                 from registers
//   column item : an 8-column x n0-row tile of A or of B (32 KB, 2D tensor copies);
//                 two CTAs per SM, so one CTA's exchanges overlap the other's arithmetic
// Row exchanges swizzle within each line (fft.cuh);
// column tiles are naturally conflict-free (a half-warp touches two whole 64-byte rows).
#include <type_traits>

#include "fft.cuh"
#include "kernels.h"
#include "tma.cuh"

namespace xsde {
namespace {

using V = float2;
using TW = float4;
constexpr int NST = 3;                        // shared-memory stages (column pass)
constexpr int kRowStages = 2;                 // (row pass)
// fields that a row mode works on
__host__ __device__ constexpr int row_fields(int mode) { return mode >= ROW_SI_START && mode <= ROW_SI_EXIT ? 1 : 2; }
constexpr uint64_t kWaitNs = 2000000000ull;    // give up on a copy after 2 s

template <int T>
__device__ __forceinline__ void line_sum2(double (&v)[2], int t, int line, double *scratch) {
    if constexpr (T <= 32) {
#pragma unroll
        for (int o = T / 2; o > 0; o >>= 1)
#pragma unroll
            for (int i = 0; i < 2; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], o);
    } else {
        constexpr int W = T / 32;
#pragma unroll
        for (int i = 0; i < 2; ++i) v[i] = warp_sum(v[i]);
        __syncthreads();
        if ((t & 31) == 0)
#pragma unroll
            for (int i = 0; i < 2; ++i) scratch[(line * W + (t >> 5)) * 2 + i] = v[i];
        __syncthreads();
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            double s = 0.0;
#pragma unroll
            for (int w = 0; w < W; ++w) s += scratch[(line * W + w) * 2 + i];
            v[i] = s;
        }
        __syncthreads();
    }
}

// on a copy that never lands: record it and drain what this CTA has in flight
__device__ void give_up(int *status, uint64_t *bars, const uint32_t *parity_next) {
    if (threadIdx.x == 0) {
        atomicOr(status, ST_TIMEOUT);
        for (int s = 0; s < NST; ++s) mbar_wait(bars + s, parity_next[s], kWaitNs);
        bulk_wait<0>();
    }
    __syncthreads();
}

// ---------------------------------------------------------------------------
// Row pass
// ---------------------------------------------------------------------------
// FIELDS: those of a work item, A and B or A alone (the semi-implicit modes).  Work
// items are small and several CTAs share an SM, each with one item in work and one
// on its way.  What bounds the pass is shared memory (L1/TEX 73 % busy, ~250 bytes a
// point of a copy engine's writes, exchanges and tables) next to issue (57 %) and
// DRAM (41 %); small CTAs wait for less at each barrier, spread a small field over
// the SMs, and leave through the registers.  64 x 512^2: 165 -> 144 us a pass against
// one CTA an SM with 64 KB items and bulk stores; one 512^2: 14.6 -> 10.1 us; five
// CTAs (96 registers, tables read through L1) 174 us.
template <int N1, int FIELDS> struct RowTma {
    static constexpr int E = 8;
    static constexpr int T = N1 / E;
    static constexpr int THREADS = FIELDS == 2 && N1 <= 512 ? 128 : 256;
    static constexpr int ROWS = THREADS / T;
    static constexpr int CTAS_PER_SM = (FIELDS == 2 ? 512 : 768) / THREADS;
    static constexpr size_t ITEM = (size_t)FIELDS * ROWS * N1 * sizeof(V);
    static constexpr size_t SCRATCH = (size_t)ROWS * (T / 32 + 1) * 2 * sizeof(double);
    static constexpr size_t SMEM = kRowStages * ITEM + (size_t)N1 * sizeof(TW) + (size_t)2 * N1 * sizeof(V) + SCRATCH +
                                   kRowStages * sizeof(uint64_t);
    static_assert(CTAS_PER_SM * (SMEM + 1024) <= 233472, "shared memory per SM");
};

// SAMPLE: this pass writes a sample; NOISE: the problem has Wiener noise.  Both
// are template flags so the common pass carries neither the sampling code nor the
// generator.
template <int N1, int MODE, bool SAMPLE, bool NOISE>
__global__ void __launch_bounds__(RowTma<N1, row_fields(MODE)>::THREADS, RowTma<N1, row_fields(MODE)>::CTAS_PER_SM)
    row_pass_tma_kernel(const Params2D<float> p) {
    constexpr int F = row_fields(MODE);
    using Cfg = RowTma<N1, F>;
    constexpr int E = Cfg::E, T = Cfg::T, ROWS = Cfg::ROWS, NST = kRowStages;
    constexpr bool IN_B = MODE == ROW_STAGE2 || MODE == ROW_STEADY || MODE == ROW_EPILOGUE;   // reads B too
    constexpr bool OUT_B = F == 2 && MODE != ROW_EPILOGUE;                                    // writes B too
    constexpr bool REAL_IN = MODE == ROW_PROLOGUE || MODE == ROW_SI_START;
    constexpr bool REAL_OUT = MODE == ROW_EPILOGUE || MODE == ROW_SI_EXIT;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    V *bufs = reinterpret_cast<V *>(smem_raw);
    TW *tw_s = reinterpret_cast<TW *>(smem_raw + NST * Cfg::ITEM);
    V *e1_s = reinterpret_cast<V *>(tw_s + N1);
    double *scratch = reinterpret_cast<double *>(e1_s + 2 * N1);
    uint64_t *bars = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(scratch) + Cfg::SCRATCH);

    const int tid = threadIdx.x;
    const int line = tid / T, t = tid - line * T;
    const int64_t nitems = p.npaths * (int64_t)p.n0 / ROWS;
    const int64_t mine = nitems > blockIdx.x ? (nitems - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    constexpr uint32_t line_bytes = (uint32_t)(N1 * sizeof(V)), vec_bytes = ROWS * line_bytes;

    // the paired twiddles as (c, s) and (c eps, s eps) halves in tw_s's N1 entries.
    // Lines of 64 points have one twiddled stage, where compensated twiddles (hi, lo)
    // both ways cost little: they keep the generic pass's transforms, and the
    // accuracy that small lattices are held to point by point
    constexpr bool PAIRED = N1 > 64;
    float2 *tw_hi = reinterpret_cast<float2 *>(tw_s), *tw_lo = tw_hi + N1;
    stage_paired(tw_hi, tw_lo, PAIRED ? p.tw1p : p.tw1, N1, tid, blockDim.x);
    if constexpr (!REAL_OUT)
        for (int i = tid; i < 2 * N1; i += blockDim.x) e1_s[i] = p.E1[i];
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) mbar_init(bars + s, 1);
        fence_barrier_init();
    }
    __syncthreads();
    // the tables above are constants; the fields are the previous pass's output
    grid_launch_dependents();
    grid_dependency_wait();

    auto issue_load = [&](int64_t k) {   // item k of this CTA into stage k % NST; warp 0, a copy a lane
        const int s = (int)(k % NST);
        const int64_t row0 = (blockIdx.x + k * gridDim.x) * ROWS;
        V *dst = bufs + (size_t)s * F * ROWS * N1;
        // (bounds-checking build: a copy past the fields is skipped, the stage
        // completes without bytes)
        const bool inside = XSDE_IN(row0 + ROWS - 1, p.npaths * (int64_t)p.n0, p.status);
        if (tid == 0) {
            if (inside) mbar_arrive_expect_tx(bars + s, IN_B ? 2 * vec_bytes : vec_bytes);
            else mbar_arrive(bars + s);
        }
        __syncwarp();
        if (!inside) return;
        if constexpr (F == 1) {
            if (tid == 0) bulk_load(dst, p.A + row0 * N1, vec_bytes, bars + s);
        } else {
            static_assert(2 * ROWS <= 32, "a copy a lane");
            const int r = tid >> 1;
            if (r < ROWS && (IN_B || !(tid & 1)))
                bulk_load(dst + tid * N1, ((tid & 1) ? p.B : p.A) + (row0 + r) * N1, line_bytes, bars + s);
        }
    };
    if (tid < 32)
        for (int64_t k = 0; k < NST && k < mine; ++k) issue_load(k);

    const float gdt = p.lt.gdt;
    const float sixth = 1.0f / 6.0f, third = 1.0f / 3.0f, half = 0.5f;
    const bool vtime = p.lt.pot == PM_TABLE && p.lt.V_nt > 1;
    const PairedTwiddles tw{tw_hi, tw_lo};
    const ExchangeLayout<V, F> L{};
    // a line's exchanges involve only its own T threads: one warp, or a named
    // barrier per line (ids 1..ROWS), so the lines of an item drift apart and
    // one line's arithmetic overlaps another's exchanges
    using LineSync = std::conditional_t<(T <= 32), SyncWarp, SyncNamed>;
    LineSync sync{};
    if constexpr (T > 32) sync = SyncNamed{1 + line, T};

    for (int64_t k = 0; k < mine; ++k) {
        const int s = (int)(k % NST);
        // every thread waits for the stage; the CTA gives up together if any timed out
        const bool landed = mbar_wait(bars + s, (uint32_t)((k / NST) & 1), kWaitNs);
        if (!__syncthreads_and(landed)) {
            if (tid == 0) {
                atomicOr(p.status, ST_TIMEOUT);
                // the items loaded and not yet waited for
                for (int64_t q = k; q < k + NST && q < mine; ++q)
                    mbar_wait(bars + q % NST, (uint32_t)((q / NST) & 1), kWaitNs);
            }
            __syncthreads();
            return;
        }
        const int64_t row0 = (blockIdx.x + k * gridDim.x) * ROWS;
        const int64_t row = row0 + line;
        const int64_t path = row / p.n0;
        const int i0 = (int)(row - path * p.n0);
        const uint32_t gp = (uint32_t)(p.lt.path_offset + path);
        // a line's A and B lie side by side: its exchanges use both as one buffer
        V *lineA = bufs + (size_t)s * F * ROWS * N1 + line * F * N1;
        V *lineB = F == 2 ? lineA + N1 : lineA;
        V *sm[F];
        sm[0] = lineA;
        if constexpr (F == 2) sm[1] = lineB;

        // 3D lattices: line i0 of a path is the point pair (i0 / nmid, i0 % nmid)
        const int la = p.ndim == 3 ? i0 / p.nmid : i0;
        const int lb = p.ndim == 3 ? i0 - la * p.nmid : 0;
        // the potential of potential() written out per dimension (no indexed
        // coordinate array, which a run-time dimension count would put in
        // local memory)
        auto pot = [&](int m, uint64_t gs) -> float {
            const int i1 = t + m * T;
            if (p.lt.pot == PM_HARMONIC) {
                const float xa = p.lt.xmin[0] + (float)la * p.lt.dx[0];
                const float xb = p.lt.xmin[1] + (float)(p.ndim == 3 ? lb : i1) * p.lt.dx[1];
                float v = 0.0f;
                v += p.lt.hw2[0] * xa * xa;
                v += p.lt.hw2[1] * xb * xb;
                if (p.ndim == 3) {
                    const float xc = p.lt.xmin[2] + (float)i1 * p.lt.dx[2];
                    v += p.lt.hw2[2] * xc * xc;
                }
                return v;
            }
            if (p.lt.pot == PM_TABLE) {
                int64_t r = p.lt.V_nt > 1 ? (int64_t)gs : 0;
                if (r >= p.lt.V_nt) r = p.lt.V_nt - 1;
                return p.lt.V[r * p.lt.npts + (int64_t)i0 * N1 + i1];
            }
            return 0.0f;
        };
        float Vst[E];
#pragma unroll
        for (int m = 0; m < E; ++m) Vst[m] = vtime ? 0.0f : pot(m, 0);
        auto potv = [&](int m, uint64_t gs) -> float { return vtime ? pot(m, gs) : Vst[m]; };
        // the noise of step sg comes from p.Z (kept by the pass that drew it), read
        // ahead of the transforms; ROW_STEADY draws and keeps that of step sg + 1,
        // ROW_PROLOGUE that of step sg
        V xi[NOISE ? E : 1];
        auto draw = [&](uint64_t gs) {
            if constexpr (NOISE)
                draw_points<float, E>(p.lt, gp, (uint32_t)gs, [&](int m) { return (uint32_t)(i0 * N1 + t + m * T); }, xi);
        };
        auto keep = [&]() {
            if constexpr (NOISE)
                if (p.Z)
#pragma unroll
                    for (int m = 0; m < E; ++m) store_noise(p.Z, p.lt.noise, row * N1 + t + m * T, xi[m]);
        };
        if constexpr (NOISE) {
            if constexpr (IN_B) {
                if (p.Z)
#pragma unroll
                    for (int m = 0; m < E; ++m) xi[m] = load_noise(p.Z, p.lt.noise, row * N1 + t + m * T);
                else draw(p.sg);
            } else if constexpr (MODE == ROW_PROLOGUE || MODE == ROW_SI_STEP) {
                draw(p.sg);
                if constexpr (MODE == ROW_PROLOGUE) keep();
            }
        }
        auto pterm = [&](int m, uint64_t gs) -> PointTerm<float> {
            if constexpr (NOISE) {
                return noisy_term(p.lt, potv(m, gs), xi[m]);
            } else {
                PointTerm<float> pt;
                pt.dtV = p.lt.dt * potv(m, gs);
                pt.na = make_float2(0.0f, 0.0f);
                return pt;
            }
        };

        V x[F][E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            x[0][m] = lineA[t + m * T];
            if constexpr (IN_B) x[1][m] = lineB[t + m * T];
        }
        sync();   // the line's natural-order reads complete before swizzled exchanges
        if constexpr (!REAL_IN) {
            if constexpr (PAIRED) fftp_bwd<N1, E, F>(x, t, sm, L, sync, tw);
            else fft<N1, E, +1, F>(x, t, sm, L, sync, tw);
        }
        // local terms of the sample of the real-space field x[0] at global step gs
        auto sample_local = [&](uint64_t gs) {
            MomentSums acc(p.sm.g);
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const float m2 = cabs2(x[0][m]);
                acc.add(m2, potv(m, gs));
                if ((p.sm.which & (MOM_MOD2 | MOM_MOD4)) && p.sm.per_point &&
                    XSDE_IN((int64_t)p.sample_slot * p.lt.npts + (int64_t)i0 * N1 + t + m * T,
                            p.sm.nsamp * p.lt.npts, p.status)) {
                    double *pp = p.sm.per_point + 2 * ((int64_t)p.sample_slot * p.lt.npts + (int64_t)i0 * N1 + t + m * T);
                    const double d = (double)m2;
                    atomicAdd(pp, d * p.sm.inv_paths);
                    atomicAdd(pp + 1, d * d * p.sm.inv_paths);
                }
            }
            double sum[2] = {acc.norm, acc.energy};
            line_sum2<T>(sum, t, line, scratch);
            if (t == 0) {
                if ((p.sm.which & (MOM_NORM | MOM_ENERGY)) && p.sm.per_path &&
                    XSDE_IN((int64_t)p.sample_slot * p.npaths + path, p.sm.nsamp * p.npaths, p.status)) {
                    double *pq = p.sm.per_path + 2 * ((int64_t)p.sample_slot * p.npaths + path);
                    atomicAdd(pq, sum[0] * p.sm.dV);
                    atomicAdd(pq + 1, sum[1] * p.sm.dV);
                }
                if (!isfinite(sum[0])) atomicOr(p.status, ST_NONFINITE);
            }
        };
        if constexpr (MODE == ROW_STAGE2) {
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const PointTerm<float> pt = pterm(m, p.sg);
                const V aI = x[0][m], k1 = x[1][m];
                const V k2 = apply_N(caxpy(aI, half, k1), pt, gdt);
                const V k3 = apply_N(caxpy(aI, half, k2), pt, gdt);
                x[0][m] = cadd(aI, k3);
                x[1][m] = caxpy(caxpy(caxpy(aI, sixth, k1), third, k2), third, k3);
            }
        } else if constexpr (MODE == ROW_SI_STEP) {
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const PointTerm<float> pt = pterm(m, p.sg);
                const V aI = x[0][m];
                V mid = aI;
#pragma unroll
                for (int it = 0; it < 3; ++it) mid = caxpy(aI, half, apply_N(mid, pt, gdt));
                x[0][m] = make_float2(2.0f * mid.x - aI.x, 2.0f * mid.y - aI.y);
            }
        } else {
            if constexpr (IN_B) {
#pragma unroll
                for (int m = 0; m < E; ++m) x[0][m] = caxpy(x[1][m], sixth, apply_N(x[0][m], pterm(m, p.sg), gdt));
            }
            if constexpr (SAMPLE) sample_local(MODE == ROW_STEADY ? p.sg + 1 : p.sg);
            if constexpr (MODE == ROW_STEADY) {
                draw(p.sg + 1);
                keep();
            }
            if constexpr (OUT_B) {
#pragma unroll
                for (int m = 0; m < E; ++m)
                    x[1][m] = apply_N(x[0][m], pterm(m, MODE == ROW_STEADY ? p.sg + 1 : p.sg), gdt);
            }
        }
        // results leave from the registers (a warp writes 256 contiguous bytes), past
        // shared memory, which is the busiest unit of this pass
        V *outA = p.A + row * N1, *outB = p.B + row * N1;
        const bool inside = XSDE_IN(row0 + ROWS - 1, p.npaths * (int64_t)p.n0, p.status);
        if constexpr (REAL_OUT) {
            if (inside)
#pragma unroll
                for (int m = 0; m < E; ++m) outA[t + m * T] = x[0][m];
        } else {
            if constexpr (PAIRED) fftp_fwd<N1, E, F>(x, t, sm, L, sync, tw);
            else fft<N1, E, -1, F>(x, t, sm, L, sync, tw);
            // the dimension-1 factor of exp(L dt/2) (hi/lo: a factor whose FP32
            // rounding misses its modulus by ~6e-8 would scale the populated modes
            // by that at every step)
            if (inside)
#pragma unroll
                for (int m = 0; m < E; ++m) {
                    const int j = t + m * T;
                    const V eh = e1_s[j], el = e1_s[N1 + j];
                    outA[j] = cmul_hilo(x[0][m], eh, el);
                    if constexpr (F == 2) outB[j] = cmul_hilo(x[1][m], eh, el);
                }
        }
        // the stage goes back to the copy engine (async proxy)
        if (k + NST < mine) {
            fence_proxy_async();
            __syncthreads();
            if (tid < 32) issue_load(k + NST);
        }
    }
}

// ---------------------------------------------------------------------------
// Column pass
// ---------------------------------------------------------------------------
template <int N0> struct ColTma {
    static constexpr int C = COL_TMA_C;                   // 64-byte row segments
    static constexpr int E = N0 >= 512 ? 16 : 8;
    static constexpr int T = N0 / E;                      // threads per column
    // independent CTAs per SM overlap their phases: 16 warps per SM
    static constexpr int CTAS_PER_SM = 512 / (C * T);
    static constexpr int THREADS = C * T;
    static constexpr int BOXR = N0 < 256 ? N0 : 256;      // tensor-copy box rows
    static constexpr size_t ITEM = (size_t)N0 * C * sizeof(V);
    static constexpr size_t SMEM = NST * ITEM + (size_t)N0 * sizeof(TW) + (size_t)2 * N0 * sizeof(V) +
                                   (THREADS / 32 + 1) * sizeof(double) + NST * sizeof(uint64_t);
};

// TRIG: dimension 0 is a cosine / sine dimension (XMDS2 Sec. 2.1): rows are
// taken from the tile in the even-odd order of the DCT-II's evaluation by an
// N0-point FFT (slot s <- row 2s below N0/2, row 2 N0-1-2s above; odd rows
// negated for the sine basis) and one exchange pairs k with N0-k for
// U_k = A_k V_k + B_k V_{N0-k} (A in E0, B in p.B0, read through L1)
template <int N0, bool TRIG = false>
__global__ void __launch_bounds__(ColTma<N0>::THREADS, ColTma<N0>::CTAS_PER_SM)
    col_pass_tma_kernel(const Params2D<float> p, const __grid_constant__ CUtensorMap mapA,
                        const __grid_constant__ CUtensorMap mapB) {
    using Cfg = ColTma<N0>;
    constexpr int C = Cfg::C, E = Cfg::E, T = Cfg::T, BOXR = Cfg::BOXR;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    V *bufs = reinterpret_cast<V *>(smem_raw);
    TW *tw_s = reinterpret_cast<TW *>(smem_raw + NST * Cfg::ITEM);
    V *e0_s = reinterpret_cast<V *>(tw_s + N0);
    double *scratch = reinterpret_cast<double *>(e0_s + 2 * N0);
    uint64_t *bars = reinterpret_cast<uint64_t *>(scratch + Cfg::THREADS / 32 + 1);

    const int tid = threadIdx.x;
    const int c = tid % C, t = tid / C;
    const int tiles = p.n1 / C;
    // two fields (A, B) per tile, or A alone for the semi-implicit scheme
    const int nvec = p.single_field ? 1 : 2;
    const int64_t nitems = p.npaths * (int64_t)tiles * nvec;
    const int64_t mine = nitems > blockIdx.x ? (nitems - 1 - blockIdx.x) / gridDim.x + 1 : 0;

    for (int i = tid; i < N0; i += blockDim.x) {
        tw_s[i] = p.tw0[i];
        e0_s[i] = p.E0[i];
        e0_s[N0 + i] = p.E0[N0 + i];
    }
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) mbar_init(bars + s, 1);
        fence_barrier_init();
    }
    __syncthreads();
    // the tables above are constants; the fields are the previous pass's output
    grid_launch_dependents();
    grid_dependency_wait();

    // item -> (vector, path, column tile)
    auto decode = [&](int64_t k, int &vec, int64_t &path, int &tile) {
        const int64_t it = blockIdx.x + k * gridDim.x;
        vec = nvec == 2 ? (int)(it & 1) : 0;
        const int64_t rest = nvec == 2 ? it >> 1 : it;
        path = rest / tiles;
        tile = (int)(rest - path * tiles);
    };
    auto issue_load = [&](int64_t k) {
        int vec, tile;
        int64_t path;
        decode(k, vec, path, tile);
        const int s = (int)(k % NST);
        V *dst = bufs + (size_t)s * N0 * C;
        const CUtensorMap *map = vec ? &mapB : &mapA;
        // (bounds-checking build: a tile past the field is skipped, the stage
        // completes without bytes)
        if (!XSDE_IN(tile * C + C - 1, p.n1, p.status) || !XSDE_IN(path, p.npaths, p.status)) {
            mbar_arrive(bars + s);
            return;
        }
        mbar_arrive_expect_tx(bars + s, (uint32_t)Cfg::ITEM);
#pragma unroll
        for (int b = 0; b < N0 / BOXR; ++b)
            tma_load_2d(dst + (size_t)b * BOXR * C, map, tile * C, (int)(path * N0 + b * BOXR), bars + s);
    };
    if (tid == 0)
        for (int64_t k = 0; k < NST - 1 && k < mine; ++k) issue_load(k);

    const TwiddleTable<TW> tw{tw_s};
    const ColumnTile<C> L{c};
    const SyncBlock sync{};
    const bool sample = p.sample_slot >= 0;

    for (int64_t k = 0; k < mine; ++k) {
        const int s = (int)(k % NST);
        // every thread waits for the stage; the CTA gives up together if any timed out
        const bool landed = mbar_wait(bars + s, (uint32_t)((k / NST) & 1), kWaitNs);
        if (!__syncthreads_and(landed)) {
            uint32_t par[NST];
            for (int q = 0; q < NST; ++q) par[q] = (uint32_t)(((k + (q - s + NST) % NST) / NST) & 1);
            give_up(p.status, bars, par);
            return;
        }
        int vec, tile;
        int64_t path;
        decode(k, vec, path, tile);
        V *tileb = bufs + (size_t)s * N0 * C;
        V *const sm1[1] = {tileb};

        const bool odd_neg = TRIG && p.basis0 == 2;
        auto row_of = [&](int j) -> int { return !TRIG ? j : (j < N0 / 2 ? 2 * j : 2 * N0 - 1 - 2 * j); };
        V x[1][E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int j = t + m * T;
            x[0][m] = tileb[row_of(j) * C + c];
            if (odd_neg && j >= N0 / 2) x[0][m] = mk<V>(-x[0][m].x, -x[0][m].y);
        }
        __syncthreads();
        fft<N0, E, -1, 1>(x, t, sm1, L, sync, tw);
        V xq[E];   // partners V_{N0-k} (TRIG)
        if constexpr (TRIG) {
#pragma unroll
            for (int m = 0; m < E; ++m) tileb[L(t + m * T)] = x[0][m];
            __syncthreads();
#pragma unroll
            for (int m = 0; m < E; ++m) xq[m] = tileb[L((N0 - t - m * T) & (N0 - 1))];
            __syncthreads();
        }
        if (sample && vec == 0) {
            // kinetic energy of a_n: sum_k Re(i L(k)) |F psi|^2 dV/(n0 n1); the
            // dimension-1 factor of exp(L dt/2) already applied is divided out
            const int col = tile * C + c;
            const int k1i = col < p.n1 / 2 ? col : col - p.n1;
            const double k1 = p.sm.kscale[1] * k1i;
            const double w = 1.0 / (double)cabs2(p.E1[col]);
            double sacc = 0.0;
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const int kj = t + m * T;
                if constexpr (TRIG) {
                    // cosine spectrum from the pair, Parseval weight 2 but at k = 0;
                    // sine mode N0-1-k sits at k
                    // (in the field's precision: the sum is accumulated in FP64)
                    float sn, cs;
                    sincospif(-(float)kj / (2.0f * N0), &sn, &cs);
                    const float xr = 0.5f * (cs * (x[0][m].x + xq[m].x) - sn * (x[0][m].y - xq[m].y));
                    const float xi = 0.5f * (cs * (x[0][m].y + xq[m].y) + sn * (x[0][m].x - xq[m].x));
                    const double k0 = p.sm.kscale[0] * (p.basis0 == 1 ? kj : N0 - kj);
                    sacc += (kj == 0 ? 1.0 : 2.0) * (p.sm.h0 + p.sm.h2 * (k0 * k0 + k1 * k1)) *
                            (double)(xr * xr + xi * xi);
                } else {
                    const double k0 = p.sm.kscale[0] * (kj < N0 / 2 ? kj : kj - N0);
                    sacc += (p.sm.h0 + p.sm.h2 * (k0 * k0 + k1 * k1)) * (double)cabs2(x[0][m]);
                }
            }
            sacc = warp_sum(sacc * w);
            if ((tid & 31) == 0) scratch[tid >> 5] = sacc;
            __syncthreads();
            if (tid == 0) {
                double tot = 0.0;
                for (int q = 0; q < Cfg::THREADS / 32; ++q) tot += scratch[q];
                if ((p.sm.which & (MOM_NORM | MOM_ENERGY)) && p.sm.per_path &&
                    XSDE_IN((int64_t)p.sample_slot * p.npaths + path, p.sm.nsamp * p.npaths, p.status))
                    atomicAdd(p.sm.per_path + 2 * ((int64_t)p.sample_slot * p.npaths + path) + 1,
                              tot * p.sm.dV / ((double)N0 * p.n1));
            }
            __syncthreads();
        }
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int j = t + m * T;
            if constexpr (TRIG)
                x[0][m] = cadd(cmul_hilo(x[0][m], e0_s[j], e0_s[N0 + j]),
                               cmul_hilo(xq[m], __ldg(p.B0 + j), __ldg(p.B0 + N0 + j)));
            else
                x[0][m] = cmul_hilo(x[0][m], e0_s[j], e0_s[N0 + j]);
        }
        fft<N0, E, +1, 1>(x, t, sm1, L, sync, tw);
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int j = t + m * T;
            tileb[row_of(j) * C + c] = (odd_neg && j >= N0 / 2) ? mk<V>(-x[0][m].x, -x[0][m].y) : x[0][m];
        }
        fence_proxy_async();
        __syncthreads();
        if (tid == 0) {
            const CUtensorMap *map = vec ? &mapB : &mapA;
            if (XSDE_IN(tile * C + C - 1, p.n1, p.status) && XSDE_IN(path, p.npaths, p.status))
#pragma unroll
                for (int b = 0; b < N0 / BOXR; ++b)
                    tma_store_2d(map, tile * C, (int)(path * N0 + b * BOXR), tileb + (size_t)b * BOXR * C);
            bulk_commit();
            if (k + NST - 1 < mine) {
                bulk_wait_read<1>();
                issue_load(k + NST - 1);
            }
        }
    }
    if (tid == 0) bulk_wait<0>();
}

template <int N1, int MODE, bool SAMPLE, bool NOISE>
cudaError_t row_tma_launch(const Params2D<float> &p, int num_sms, cudaStream_t s) {
    using Cfg = RowTma<N1, row_fields(MODE)>;
    auto kern = row_pass_tma_kernel<N1, MODE, SAMPLE, NOISE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t items = p.npaths * (int64_t)p.n0 / Cfg::ROWS, want = (int64_t)num_sms * Cfg::CTAS_PER_SM;
    const int g = (int)(items < want ? items : want);
    return launch_dependent(kern, g, Cfg::THREADS, Cfg::SMEM, s, p);
}

template <int N0>
cudaError_t col_tma_launch(const Params2D<float> &p, const CUtensorMap &a, const CUtensorMap &b, int grid,
                           cudaStream_t s) {
    using Cfg = ColTma<N0>;
    auto kern = p.basis0 ? col_pass_tma_kernel<N0, true> : col_pass_tma_kernel<N0, false>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t items = p.npaths * (int64_t)(p.n1 / Cfg::C) * (p.single_field ? 1 : 2);
    const int64_t want = (int64_t)grid * Cfg::CTAS_PER_SM;
    const int g = (int)(items < want ? items : want);
    return launch_dependent(kern, g, Cfg::THREADS, Cfg::SMEM, s, p, a, b);
}

}  // namespace

bool tma_row_supported(int n1) { return n1 == 64 || n1 == 128 || n1 == 256 || n1 == 512 || n1 == 1024; }
bool tma_col_supported(int n0) { return n0 == 128 || n0 == 256 || n0 == 512; }

template <int N1> cudaError_t row_tma_dispatch(int mode, const Params2D<float> &p, int num_sms, cudaStream_t s) {
    const bool noise = p.lt.noise != NM_NONE, sample = p.sample_slot >= 0;
    // (mode, samples, uses noise): the instantiated combinations
    switch (mode) {
        case ROW_STAGE2:
            return noise ? row_tma_launch<N1, ROW_STAGE2, false, true>(p, num_sms, s)
                         : row_tma_launch<N1, ROW_STAGE2, false, false>(p, num_sms, s);
        case ROW_STEADY:
            if (sample)
                return noise ? row_tma_launch<N1, ROW_STEADY, true, true>(p, num_sms, s)
                             : row_tma_launch<N1, ROW_STEADY, true, false>(p, num_sms, s);
            return noise ? row_tma_launch<N1, ROW_STEADY, false, true>(p, num_sms, s)
                         : row_tma_launch<N1, ROW_STEADY, false, false>(p, num_sms, s);
        case ROW_PROLOGUE:
            if (sample)
                return noise ? row_tma_launch<N1, ROW_PROLOGUE, true, true>(p, num_sms, s)
                             : row_tma_launch<N1, ROW_PROLOGUE, true, false>(p, num_sms, s);
            return noise ? row_tma_launch<N1, ROW_PROLOGUE, false, true>(p, num_sms, s)
                         : row_tma_launch<N1, ROW_PROLOGUE, false, false>(p, num_sms, s);
        case ROW_EPILOGUE:
            return noise ? row_tma_launch<N1, ROW_EPILOGUE, false, true>(p, num_sms, s)
                         : row_tma_launch<N1, ROW_EPILOGUE, false, false>(p, num_sms, s);
        case ROW_SI_START: return row_tma_launch<N1, ROW_SI_START, false, false>(p, num_sms, s);
        case ROW_SI_STEP:
            return noise ? row_tma_launch<N1, ROW_SI_STEP, false, true>(p, num_sms, s)
                         : row_tma_launch<N1, ROW_SI_STEP, false, false>(p, num_sms, s);
        case ROW_SI_EXIT:
            return sample ? row_tma_launch<N1, ROW_SI_EXIT, true, false>(p, num_sms, s)
                          : row_tma_launch<N1, ROW_SI_EXIT, false, false>(p, num_sms, s);
        default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_row_pass_tma(int mode, const Params2D<float> &p, int num_sms, cudaStream_t s) {
    switch (p.n1) {
        case 64: return row_tma_dispatch<64>(mode, p, num_sms, s);
        case 128: return row_tma_dispatch<128>(mode, p, num_sms, s);
        case 256: return row_tma_dispatch<256>(mode, p, num_sms, s);
        case 512: return row_tma_dispatch<512>(mode, p, num_sms, s);
        case 1024: return row_tma_dispatch<1024>(mode, p, num_sms, s);
        default: return cudaErrorInvalidValue;
    }
}
int64_t tma_row_lines(int n1, int fields) { return (fields == 2 && n1 <= 512 ? 128 : 256) / (n1 / 8); }

cudaError_t launch_col_pass_tma(const Params2D<float> &p, const CUtensorMap &a, const CUtensorMap &b, int grid,
                                cudaStream_t s) {
    switch (p.n0) {
        case 128: return col_tma_launch<128>(p, a, b, grid, s);
        case 256: return col_tma_launch<256>(p, a, b, grid, s);
        case 512: return col_tma_launch<512>(p, a, b, grid, s);
        default: return cudaErrorInvalidValue;
    }
}

size_t col_tma_box_rows(int n0) { return n0 < 256 ? (size_t)n0 : 256; }

}  // namespace xsde
