// rk4ip_2d_warp.cu -- the complex64 column pass with warp-synchronous transforms.
//
// Same arithmetic as rk4ip_2d.cu (XMDS2 Sec. 2.6: exp(L dt/2) applied in
// Fourier space between real-space RK4 stages; Sec. 2.2: the transform of a
// tensor-product lattice factorises per dimension), organised so that no
// transform waits on another warp:
//   column pass : 8-column tiles of A or B (64-byte rows, 64-byte TMA swizzle)
//                 stream through a ring of shared-memory stages; each warp owns
//                 two (or four) columns of the tile and transforms them with the
//                 two-stage plan of fft2.cuh, exchanging in place inside its own
//                 columns.  The last warp to finish a tile stores it and refills
//                 the stage; several groups of warps per SM keep it busy while one
//                 of them waits.
//
// Every wait is bounded by the global timer; a wait that runs out records
// ST_TIMEOUT, lets the group's other warps stop, waits (bounded) for the group's
// copies in flight and returns.
#include <type_traits>

#include "fft2.cuh"
#include "kernels.h"
#include "tma.cuh"

namespace xsde {
namespace {

using V = float2;
using TW = float4;
constexpr uint64_t kWaitNs = 2000000000ull;   // give up on a copy after 2 s

// Wait for phase `parity` of `bar`; false once `abort_flag` is set or the
// time limit passes.
__device__ __forceinline__ bool wait_or_abort(uint64_t *bar, uint32_t parity, const volatile int *abort_flag) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = global_timer_ns();
    while (!mbar_try_wait(bar, parity)) {
        if (*abort_flag) return false;
        if (global_timer_ns() - t0 > kWaitNs) return false;
    }
    return true;
}

// ---------------------------------------------------------------------------
// Column pass
// ---------------------------------------------------------------------------
enum { COLW_PLAIN = 0, COLW_TRIG = 1, COLW_CONV = 2 };   // kinds of column pass
template <int N0, bool SPREAD, bool TRIG> struct ColW {
    static constexpr int E = N0 >= 256 ? N0 / 16 : N0 == 128 ? 16 : 8;   // points per lane: 32 / 16 / 16 / 8
    static constexpr int P = N0 / E;                           // lanes per column: 16 / 16 / 8 / 8
    static constexpr int C = WARP_COL_C;                       // tile columns (64-byte rows)
    static constexpr int CPW = 32 / P;                         // columns per warp
    static constexpr int NW = C / CPW;                         // warps per tile: 4 / 4 / 2 / 2
    // A CTA is GROUPS independent groups of NW warps, each with its own stages, that
    // share one copy of the tables (the room for them is what held an SM to 8 warps
    // at 512 points): 12 warps at 167 registers, 16 at 128 for the shorter columns.
    // 64 x 512^2: 136 -> 120 us; 16 warps with one stage each 163 us.  SPREAD: one
    // group, for fields of few tiles.
    // (TRIG holds the partner values too: 8 to 12 warps)
    static constexpr int GROUPS = SPREAD ? 1 : TRIG ? (N0 == 256 ? 3 : 6) : N0 == 512 ? 3 : N0 == 256 ? 4 : 8;
    static constexpr int THREADS = GROUPS * NW * 32;
    static constexpr int NST = N0 == 512 ? 2 : 3;        // shared-memory stages of a group
    static constexpr int BOXR = N0 < 256 ? N0 : 256;           // tensor-copy box rows
    static constexpr size_t TILE = (size_t)N0 * C * sizeof(V); // 32 / 16 / 8 / 4 KB
    static constexpr int NTW = warp_fft_table_size<N0, E>();
    // (512 points: a compact (c, s) copy of the twiddles for the forward, NTW float2)
    static constexpr size_t TWF = N0 > 256 ? NTW * sizeof(float2) : 0;
    static constexpr size_t SMEM = 1024 + GROUPS * NST * TILE + NTW * sizeof(TW) + 2 * N0 * sizeof(V) + TWF +
                                   GROUPS * (NST * (sizeof(uint64_t) + sizeof(long long) + sizeof(int)) + 16);
    static_assert(SMEM + 1024 <= 233472, "shared memory per SM");
};

// The stage ring has no producer warp: thread 0 fills the first stages, and
// the last warp to finish a tile (an arrival count per stage) stores it and
// refills its stage with the tile NST items later.  A bulk store's completion
// is tracked per thread, so that warp also waits until its store has read the
// stage before the load reuses it.
// TRIG: dimension 0 is a cosine / sine dimension (XMDS2 Sec. 2.1): rows are
// taken from the tile in the even-odd order of the DCT-II's evaluation by an
// N0-point FFT (slot s <- row 2s below N0/2, row 2 N0-1-2s above; odd rows
// negated for the sine basis) and one exchange pairs k with N0-k for
// U_k = A_k V_k + B_k V_{N0-k} (A in E0, B in p.B0, read through L1).  16 x 256 x 512:
// 33 us a pass in the TMA column kernel, 27 us here.
// CONV: the density convolution of the non-local term, K2(k0, col) (read through L1)
// in place of E0(k0), on the one field the maps describe.
// SAMPLE: this pass writes a sample; a template flag, so that the common pass does not
// carry the sampling code (its registers are all taken).
template <int N0, bool SPREAD, int KIND, bool SAMPLE>
__global__ void __launch_bounds__(ColW<N0, SPREAD, KIND == COLW_TRIG>::THREADS, 1)
    col_pass_warp_kernel(const Params2D<float> p, const __grid_constant__ CUtensorMap mapA,
                         const __grid_constant__ CUtensorMap mapB) {
    constexpr bool TRIG = KIND == COLW_TRIG, CONV = KIND == COLW_CONV;
    using Cfg = ColW<N0, SPREAD, TRIG>;
    constexpr int E = Cfg::E, P = Cfg::P, C = Cfg::C, CPW = Cfg::CPW, NW = Cfg::NW, NST = Cfg::NST,
                  BOXR = Cfg::BOXR;
    extern __shared__ unsigned char smem_raw[];
    // tiles start on a 1024-byte boundary (the swizzle pattern repeats every 512)
    unsigned char *base = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    constexpr int GROUPS = Cfg::GROUPS, GT = NW * 32;   // groups, threads of one
    const int group = threadIdx.x / GT;
    unsigned char *tiles = base + (size_t)group * NST * Cfg::TILE;
    TW *tw_s = reinterpret_cast<TW *>(base + (size_t)GROUPS * NST * Cfg::TILE);
    V *e0_s = reinterpret_cast<V *>(tw_s + Cfg::NTW);
    float2 *twf_s = reinterpret_cast<float2 *>(e0_s + 2 * N0);          // e0_s: hi[N0] | lo[N0]
    uint64_t *full = reinterpret_cast<uint64_t *>(reinterpret_cast<unsigned char *>(twf_s) + Cfg::TWF);
    volatile long long *issued = reinterpret_cast<volatile long long *>(full + GROUPS * NST);   // last item loaded per stage
    int *done = reinterpret_cast<int *>(const_cast<long long *>(issued) + GROUPS * NST);         // warps finished per stage
    volatile int *abort_flag = done + GROUPS * NST + group;
    full += group * NST;
    issued += group * NST;
    done += group * NST;

    // (within the group)
    const int tid = threadIdx.x - group * GT, warp = tid >> 5, lane = tid & 31;
    // tiles go to the SMs in turn before they go to another group of the same SM
    const int64_t vblock = blockIdx.x + (int64_t)group * gridDim.x, vgrid = (int64_t)gridDim.x * GROUPS;
    const int tiles_per_path = p.n1 / C;
    // two fields (A, B) per tile, or A alone for the semi-implicit scheme
    const int nvec = p.single_field ? 1 : 2;
    const int64_t nitems = p.npaths * (int64_t)tiles_per_path * nvec;
    const int64_t mine = nitems > vblock ? (nitems - 1 - vblock) / vgrid + 1 : 0;

    // columns of 128 and 256 points (shared-memory-bound at 16 points a lane)
    // stage the paired twiddles as split (c, s) / (c eps, s eps) arrays, so the
    // forward reads 8 bytes a lane at an 8-byte stride; 512 keeps float4 entries
    // for the backward (one 16-byte read a twiddle) and a compact (c, s) copy
    // for the forward
    constexpr bool SPLIT = N0 <= 256;
    float2 *tw_hi = reinterpret_cast<float2 *>(tw_s), *tw_lo = tw_hi + Cfg::NTW;
    if constexpr (SPLIT) {
        stage_paired(tw_hi, tw_lo, p.tw0w, Cfg::NTW, threadIdx.x, blockDim.x);
    } else {
        for (int i = threadIdx.x; i < Cfg::NTW; i += blockDim.x) {
            const TW w = p.tw0w[i];
            tw_s[i] = w;
            twf_s[i] = make_float2(w.x, w.y);
        }
    }
    for (int i = threadIdx.x; i < 2 * N0 && !CONV; i += blockDim.x) e0_s[i] = p.E0[i];
    if (tid == 0) {
        for (int s = 0; s < NST; ++s) {
            mbar_init(full + s, 1);
            issued[s] = -1;
            done[s] = 0;
        }
        *abort_flag = 0;
        fence_barrier_init();
    }
    __syncthreads();
    // the tables above are constants; the fields are the previous pass's output
    grid_launch_dependents();
    grid_dependency_wait();

    // item -> (vector, path, column tile)
    auto decode = [&](int64_t k, int &vec, int64_t &path, int &tile) {
        const uint32_t it = (uint32_t)(vblock + k * vgrid);
        vec = nvec == 2 ? (int)(it & 1) : 0;
        const uint32_t rest = nvec == 2 ? it >> 1 : it;
        const uint32_t pth = rest / (uint32_t)tiles_per_path;
        path = pth;
        tile = (int)(rest - pth * (uint32_t)tiles_per_path);
    };
    auto issue_load = [&](int64_t k) {
        int vec, tile;
        int64_t path;
        decode(k, vec, path, tile);
        const int s = (int)(k % NST);
        unsigned char *dst = tiles + (size_t)s * Cfg::TILE;
        issued[s] = k;
        // (bounds-checking build: a tile past the field is skipped, the stage
        // completes without bytes)
        if (!XSDE_IN(tile * C + C - 1, p.n1, p.status) || !XSDE_IN(path, p.npaths, p.status)) {
            mbar_arrive(full + s);
            return;
        }
        mbar_arrive_expect_tx(full + s, (uint32_t)Cfg::TILE);
#pragma unroll
        for (int b = 0; b < N0 / BOXR; ++b)
            tma_load_2d(dst + (size_t)b * BOXR * (C * 8), vec ? &mapB : &mapA, tile * C, (int)(path * N0 + b * BOXR),
                        full + s);
    };
    auto issue_store = [&](int64_t k) {
        int vec, tile;
        int64_t path;
        decode(k, vec, path, tile);
        const unsigned char *src = tiles + (size_t)(k % NST) * Cfg::TILE;
        if (XSDE_IN(tile * C + C - 1, p.n1, p.status) && XSDE_IN(path, p.npaths, p.status))
#pragma unroll
            for (int b = 0; b < N0 / BOXR; ++b)
                tma_store_2d(vec ? &mapB : &mapA, tile * C, (int)(path * N0 + b * BOXR),
                             src + (size_t)b * BOXR * (C * 8));
        bulk_commit();
    };
    // leave on a copy that never lands: record it, stop the CTA's other warps
    // and wait (bounded) for the loads in flight and this thread's stores
    auto give_up = [&]() {
        if (lane == 0) {
            atomicOr(p.status, ST_TIMEOUT);
            *abort_flag = 1;
            for (int s = 0; s < NST; ++s) {
                const long long kk = issued[s];
                if (kk >= 0) mbar_wait(full + s, (uint32_t)((kk / NST) & 1), kWaitNs);
            }
            bulk_wait<0>();
        }
        __syncwarp();
    };
    if (tid == 0)
        for (int64_t k = 0; k < NST && k < mine; ++k) issue_load(k);

    // The warp owns columns warp * CPW .. + CPW-1.  Eight-byte shared accesses
    // are served in two 16-lane phases, so each phase must span all of the
    // warp's columns (a column's rows reach only 8 of the 16 bank pairs of a
    // swizzled 128-byte row): two columns alternate lane by lane; four columns
    // take lanes in blocks of 8 (each half-warp then holds two columns).
    const int c = CPW == 2 ? warp * 2 + (lane & 1) : warp * CPW + lane / P;
    const int t = CPW == 2 ? lane >> 1 : lane % P;
    const auto tw = [&] {
        if constexpr (SPLIT) return PairedTwiddles{tw_hi, tw_lo};
        else return TwiddleTable<TW>{tw_s};
    }();
    // the forward's twiddles: the (c, s) halves only (tw_fwd reads no more)
    const auto twf = [&] {
        if constexpr (SPLIT) return PairedTwiddles{tw_hi, tw_lo};
        else return PairedTwiddles{twf_s, twf_s};
    }();
    for (int64_t k = 0; k < mine; ++k) {
        const int s = (int)(k % NST);
        if (!wait_or_abort(full + s, (uint32_t)((k / NST) & 1), abort_flag)) {
            give_up();
            return;
        }
        int vec, tile;
        int64_t path;
        decode(k, vec, path, tile);
        unsigned char *tb = tiles + (size_t)s * Cfg::TILE;
        // element (row, c) of the tile as the 64-byte swizzle lays it out: in
        // 64-byte rows, 16-byte chunk (c / 2) ^ ((row / 2) % 4); its offset is XOR-linear
        // in the row, row_off, so an access is the lane's own offset, an XOR and a constant
        auto row_off = [](int row) -> int { return (row << 6) ^ (((row >> 1) & 3) << 4); };
        const int co = ((c >> 1) << 4) | ((c & 1) << 3);
        const int rt = row_off(t) ^ co, wt = row_off(t & 7) ^ co;
        unsigned char *const tbw = tb + 64 * E * t;
        using Slots = ColumnSlots<N0, E>;
        auto nat = [&](int m) -> V * { return reinterpret_cast<V *>(tb + rt + 64 * P * m); };   // row t + P m
        auto xw = [&](int r) -> V * {
            return reinterpret_cast<V *>(tbw + (wt ^ row_off(Slots::write_low(r))) + 64 * Slots::write_high(r));
        };
        auto xr = [&](int m) -> V * {
            return reinterpret_cast<V *>(tb + (rt ^ row_off(Slots::read_low(m))) + 64 * Slots::read_high(m));
        };
        // (TRIG) the slots t + P m below N0/2 lie at rows 2t + 2 P m, the others at
        // 2 N0 - 1 - 2 P m - 2t
        const bool odd_neg = TRIG && p.basis0 == 2;
        auto gather = [&](int m) -> V * {
            const int chunk = m < E / 2 ? (t & 3) : 3 - (t & 3);
            const int row = m < E / 2 ? 2 * t + 2 * P * m : 2 * N0 - 1 - 2 * P * m - 2 * t;
            return reinterpret_cast<V *>(tb + 64 * row + ((chunk << 4) ^ co));
        };
        V x[E];
#pragma unroll
        for (int m = 0; m < E; ++m) {
            x[m] = TRIG ? *gather(m) : *nat(m);
            if (odd_neg && m >= E / 2) x[m] = make_float2(-x[m].x, -x[m].y);
        }
        __syncwarp();
        warp_fft<N0, E, (N0 == 64)>(x, t, xw, xr, twf);
        V xq[TRIG ? E : 1];   // partners V_{N0-k}
        if constexpr (TRIG) {
#pragma unroll
            for (int m = 0; m < E; ++m) *nat(m) = x[m];
            __syncwarp();
#pragma unroll
            for (int m = 0; m < E; ++m) xq[m] = *reinterpret_cast<V *>(tb + (row_off((N0 - P * m - t) & (N0 - 1)) ^ co));
            __syncwarp();
        }
        if (SAMPLE && vec == 0) {
            // kinetic energy of a_n: sum_k Re(i L(k)) |F psi|^2 dV/(n0 n1); the
            // dimension-1 factor of exp(L dt/2) already applied is divided out
            const int col = tile * C + c;
            const int k1i = col < p.n1 / 2 ? col : col - p.n1;
            const double k1 = p.sm.kscale[1] * k1i;
            const double w = 1.0 / (double)cabs2(p.E1[col]);
            // h(k) = (h0 + h2 k1^2) + h2 ks^2 kj^2: two FP64 sums, of |X|^2 and kj^2 |X|^2
            double s0 = 0.0, s2 = 0.0;
#pragma unroll
            for (int m = 0; m < E; ++m) {
                const int kj = t + P * m;
                if constexpr (TRIG) {
                    // cosine spectrum from the pair, Parseval weight 2 but at k = 0;
                    // sine mode N0-1-k sits at k
                    // (in the field's precision: the sum is accumulated in FP64)
                    float sn, cs;
                    sincospif(-(float)kj / (2.0f * N0), &sn, &cs);
                    const float xr = 0.5f * (cs * (x[m].x + xq[m].x) - sn * (x[m].y - xq[m].y));
                    const float xi = 0.5f * (cs * (x[m].y + xq[m].y) + sn * (x[m].x - xq[m].x));
                    const int kb = p.basis0 == 1 ? kj : N0 - kj;
                    const double d = widen((kj == 0 ? 1.0f : 2.0f) * (xr * xr + xi * xi));
                    s0 += d;
                    s2 = fma(widen_whole(kb * kb), d, s2);
                } else {
                    const int kb = kj < N0 / 2 ? kj : kj - N0;
                    const double d = widen(cabs2(x[m]));
                    s0 += d;
                    s2 = fma(widen_whole(kb * kb), d, s2);
                }
            }
            double sacc = (p.sm.h0 + p.sm.h2 * k1 * k1) * s0 + p.sm.h2 * p.sm.kscale[0] * p.sm.kscale[0] * s2;
            sacc = warp_sum(sacc * w);
            if (lane == 0 && (p.sm.which & (MOM_NORM | MOM_ENERGY)) && p.sm.per_path &&
                XSDE_IN((int64_t)p.sample_slot * p.npaths + path, p.sm.nsamp * p.npaths, p.status))
                atomicAdd(p.sm.per_path + 2 * ((int64_t)p.sample_slot * p.npaths + path) + 1,
                          sacc * p.sm.dV / ((double)N0 * p.n1));
        }
#pragma unroll
        for (int m = 0; m < E; ++m) {
            const int j = t + P * m;
            if constexpr (CONV) x[m] = cmul(x[m], __ldg(p.K2 + (int64_t)j * p.n1 + tile * C + c));
            else x[m] = cmul_hilo(x[m], e0_s[j], e0_s[N0 + j]);
            if constexpr (TRIG) x[m] = cadd(x[m], cmul_hilo(xq[m], __ldg(p.B0 + j), __ldg(p.B0 + N0 + j)));
        }
        warp_ifft<N0, E>(x, t, xw, xr, tw);
#pragma unroll
        for (int m = 0; m < E; ++m) {
            if (odd_neg && m >= E / 2) x[m] = make_float2(-x[m].x, -x[m].y);
            *(TRIG ? gather(m) : nat(m)) = x[m];
        }
        // the tile goes out through the tensor-memory-access unit (async proxy)
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
            __threadfence_block();
            if (atomicAdd(done + s, 1) == NW - 1) {
                // every warp has written its columns of the tile
                atomicExch(done + s, 0);
                __threadfence_block();
                issue_store(k);
                if (k + NST < mine) {
                    bulk_wait_read<0>();
                    issue_load(k + NST);
                }
            }
        }
        __syncwarp();
    }
    if (lane == 0) bulk_wait<0>();
}

template <int N0, bool SPREAD, int KIND, bool SAMPLE = false>
cudaError_t col_warp_launch_as(const Params2D<float> &p, int64_t items, const CUtensorMap &a, const CUtensorMap &b,
                               int num_sms, cudaStream_t s) {
    if constexpr (KIND != COLW_CONV && !SAMPLE)
        if (p.sample_slot >= 0) return col_warp_launch_as<N0, SPREAD, KIND, true>(p, items, a, b, num_sms, s);
    using Cfg = ColW<N0, SPREAD, KIND == COLW_TRIG>;
    auto kern = col_pass_warp_kernel<N0, SPREAD, KIND, SAMPLE>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
    if (e != cudaSuccess) return e;
    const int64_t want = SPREAD ? items : num_sms;
    return launch_dependent(kern, (int)(items < want ? items : want), Cfg::THREADS, Cfg::SMEM, s, p, a, b);
}
// few tiles are spread over the SMs, one group to a CTA
template <int N0>
cudaError_t col_warp_launch(const Params2D<float> &p, const CUtensorMap &a, const CUtensorMap &b, bool conv, int num_sms,
                            cudaStream_t s) {
    const int64_t items = p.npaths * (int64_t)(p.n1 / WARP_COL_C) * (p.single_field ? 1 : 2);
    if (conv) return col_warp_launch_as<N0, false, COLW_CONV>(p, items, a, b, num_sms, s);
    if (p.basis0) {
        if constexpr (N0 == 128 || N0 == 256) return col_warp_launch_as<N0, false, COLW_TRIG>(p, items, a, b, num_sms, s);
        else return cudaErrorInvalidValue;   // (col_pass_kind takes other passes)
    }
    return items <= 2 * (int64_t)num_sms ? col_warp_launch_as<N0, true, COLW_PLAIN>(p, items, a, b, num_sms, s)
                                         : col_warp_launch_as<N0, false, COLW_PLAIN>(p, items, a, b, num_sms, s);
}

}  // namespace

bool warp_col_supported(int n0, int64_t n1) {
    return (n0 == 64 || n0 == 128 || n0 == 256 || n0 == 512) && n1 % WARP_COL_C == 0;
}
int warp_col_elems(int n0) { return n0 >= 256 ? n0 / 16 : n0 == 128 ? 16 : 8; }
size_t warp_col_box_rows(int n0) { return n0 < 256 ? (size_t)n0 : 256; }

static cudaError_t col_pass_warp_any(const Params2D<float> &p, const CUtensorMap &a, const CUtensorMap &b, bool conv,
                                     int num_sms, cudaStream_t s) {
    switch (p.n0) {
        case 64: return col_warp_launch<64>(p, a, b, conv, num_sms, s);
        case 128: return col_warp_launch<128>(p, a, b, conv, num_sms, s);
        case 256: return col_warp_launch<256>(p, a, b, conv, num_sms, s);
        case 512: return col_warp_launch<512>(p, a, b, conv, num_sms, s);
        default: return cudaErrorInvalidValue;
    }
}
cudaError_t launch_col_pass_warp(const Params2D<float> &p, const CUtensorMap &a, const CUtensorMap &b, int num_sms,
                                 cudaStream_t s) {
    if (!p.tw0w || (p.basis0 && !p.B0)) return cudaErrorInvalidValue;
    return col_pass_warp_any(p, a, b, false, num_sms, s);
}
cudaError_t launch_col_conv_warp(const Params2D<float> &p, const CUtensorMap &mapC, int num_sms, cudaStream_t s) {
    if (!p.tw0w || !p.K2 || p.basis0) return cudaErrorInvalidValue;
    Params2D<float> q = p;
    q.single_field = 1;
    return col_pass_warp_any(q, mapC, mapC, true, num_sms, s);
}

}  // namespace xsde
