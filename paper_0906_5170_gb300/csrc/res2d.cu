// Resident march of the two-dimensional (TM-form) simulations: a thread-block cluster holds one
// simulation's fields in registers and advances it through a whole chunk of time steps per launch.
//
// The update is that of step2d.cu and step2d_tk.cu (McCauley et al., arXiv:0906.5170: harmonic
// source J = delta(t) f_n on S, Yee leapfrog in a medium of conductivity sigma, surface functional
// weighted by w_n = 2 dt Im g(-n dt), Eq. (1)), value for value.
//
// Layout: a thread owns a block of CX columns (16 bytes) by RB rows of u, vx, vy in registers;
// `tcols` threads cover a row band of the grid, bands are RB or RB - 1 rows high, and the bands
// are dealt to the cluster's CTAs in order, from grid row `shift` on (so that no CTA boundary parts the
// rows of a horizontal face, whose functional may cancel along it and is summed step by step in one CTA).
// The grid is a torus (closed walls are masked sites), so the first band's upper neighbour is the last
// band.  Per step
//   V: vx(r) from u(r + 1) - u(r), vy(c) from u(c + 1) - u(c)
//   U: u from vy(c) - vy(c - 1) and vx(r) - vx(r - 1)
// (sigma on u: V then U; sigma on v: U then V, run as U, (V, U), ..., V).  A thread updates vx of the row
// above and vy of the column to the left of its block as well as its own, so that one exchange per
// step is enough: the u values on the block's four edges, written to the neighbours' slots in shared
// memory.  U of the edge cells comes first, then the exchange, then U of the inner cells and the part of
// the next V that needs no neighbour, and only then the step's barrier.  A row for the next or the
// previous CTA goes by st.async, which counts its bytes on that CTA's mbarrier; only the warps of the
// band that needs it wait there.  Two buffers of slots by step parity: a neighbour writes the slots of
// step n + 2 only after the barrier that follows this thread's reads of step n.
//
// Bound by the chain of one step (slots, barrier, far rows) on small grids and by that and issue on large
// ones (16 warps of 128 registers on an SM, 45% of the issue slots); memory holds the fields only between
// launches of up to 192 steps.  Measured against the multi-step kernels, whose fields pass through memory
// every two or three steps (Gcell-updates/s): FP32 400 x 166, 640 simulations 465 -> 779; 128 x 128, 320
// simulations 734, 64 x 64, 160 simulations 514, 60 x 20, 96 simulations 155; whole FP64 plate forces 88.5 -> 8.3 ms, FP64
// 251 x 93 44.5 -> 24.6 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <utility>

#include "resident.cuh"

namespace cas {

namespace {

// A block's u depends on vx of the row above and vy of the column to the left.  RED (FP32): the thread
// updates those itself as well, from the u around its block, so that one exchange of u per step is enough.
// Without (FP64, whose arithmetic is the limit: 17 to 33% more of it lost 20%): the neighbours send vx and vy
// after V, and u after U.
template <typename R>
constexpr bool RES_RED = sizeof(R) == 4;

// 16-byte words of a thread's slots in shared memory, filled by its neighbours: a row from above (RED: u,
// else vx), u of the row below, a column from the left (RED: u, else vy), u of the column to the right;
// RED: two buffers by step parity.  And of the coefficients of its cells, in warps whose cells are not all
// of one material: vx (RED: from the row above on), vy (RED: the column to the left last), u.  Odd counts
// keep the 16-byte accesses of consecutive threads free of bank conflicts.
template <typename R, int RB>
struct Slots {
    static constexpr int CX = 16 / (int)sizeof(R), RED = RES_RED<R> ? 1 : 0;
    static constexpr int KV = (RB + CX - 1) / CX;
    static constexpr int UP = 0, DN = 1, LF = 2, RT = 2 + KV, BUF = 2 + 2 * KV;
    static constexpr int WORDS = ((1 + RED) * BUF) | 1;
    static constexpr int CVX = 0, CVY = RB + RED, CVYL = 2 * RB + RED, CU = 2 * RB + RED * (1 + KV);
    static constexpr int CWORDS = (3 * RB + RED * (1 + KV)) | 1;
};

template <typename R, int RB, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
k_res2d(const DevRes2D *__restrict__ sims, int64_t launch, int count)
{
    using V4 = Vec16<R>;
    using SL = Slots<R, RB>;
    constexpr int CX = SL::CX, KV = SL::KV;
    constexpr bool RED = RES_RED<R>;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ short slot[RES_PIECES * 32 + 1];           // entries of each piece's 32 partial sums
    __shared__ short piece[RES_PIECES];                   // the simulation's numbers of this CTA's pieces
    __shared__ __align__(8) unsigned long long mbar[4];   // rows from the previous and from the next CTA, by step parity

    const unsigned C = cluster_size(), rank = cluster_rank();
    const DevRes2D &D = sims[blockIdx.x / C];
    const DevSim2D &S = D.s;
    // the launch indices of this launch and the time steps they hold (the same for the whole cluster)
    const int64_t L0 = launch - S.s0;
    const int64_t l_lo = L0 > 1 ? L0 : 1, l_hi = L0 + count - 1;
    if (l_hi < l_lo || (l_lo - 1) * D.k + 1 > S.T) return;
    const int n_lo = (int)((l_lo - 1) * D.k + 1), n_hi = (int)min((int64_t)S.T, l_hi * D.k);
    const int cnt = n_hi - n_lo + 1;
    const bool multi = C > 1;

    const int nt = blockDim.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nx = S.nx, ny = S.ny, nb = D.nb, tcols = D.tcols;
    const unsigned N = (unsigned)nx * (unsigned)ny;
    const int b0 = (int)rank * nb / (int)C, b1 = ((int)rank + 1) * nb / (int)C;   // this CTA's bands
    const int lb = t / tcols, tc = t - lb * tcols, b = b0 + lb;
    const bool active = b < b1;
    const int y0 = active ? b * ny / nb : 0;
    const int h = active ? (b + 1) * ny / nb - y0 : RB;   // RB or RB - 1
    const int x0 = tc * CX;
    const int w = active ? min(CX, nx - x0) : CX;          // valid columns

    const unsigned mb_u = (unsigned)__cvta_generic_to_shared(&mbar[0]), mb_d = mb_u + 16;
    if (multi && t == 0) {
        // two each: the neighbour may send the rows of step i + 1 before all those of step i have landed
        // (never those of step i + 2, which wait for this CTA's answer to step i)
        for (int q = 0; q < 4; ++q) mb_init(mb_u + 8 * q, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int q = 0; q < 4; ++q) mb_expect(mb_u + 8 * q, tcols * 16);
    }

    // this thread's slots, and those its edges go to: its u row 0 to the band above, its last row to the
    // band below, its column 0 to the left, its last column to the right.  What a step needs beside the
    // fields is packed into a few registers: with the fields in registers every further value that
    // stays live through the loop costs a spill.
    V4 *const blocks = reinterpret_cast<V4 *>(dyn);
    const int own_i = t * SL::WORDS;
    unsigned cu = rank, cd = rank;   // the CTAs of the bands above and below
    auto band_slot = [&](int bb, unsigned *cta) {
        unsigned r = rank;
        if (bb < b0 || bb >= b1)   // the ends of a CTA's range meet the next and the previous CTA of the ring
            r = (bb == (b1 == nb ? 0 : b1)) ? (rank + 1 == C ? 0 : rank + 1) : (rank == 0 ? C - 1 : rank - 1);
        *cta = r;
        return ((bb - (int)r * nb / (int)C) * tcols + tc) * SL::WORDS;
    };
    const int iu = (active ? band_slot(b == 0 ? nb - 1 : b - 1, &cu) : own_i) + SL::DN;
    const int id = (active ? band_slot(b + 1 == nb ? 0 : b + 1, &cd) : own_i) + SL::UP;
    const int il = own_i + (tc == 0 ? tcols - 1 : -1) * SL::WORDS + SL::RT;
    const int ir = own_i + (tc == tcols - 1 ? 1 - tcols : 1) * SL::WORDS + SL::LF;
    unsigned pk_row = (unsigned)iu | (unsigned)id << 16, pk_col = (unsigned)(active ? il : own_i) | (unsigned)(active ? ir : own_i) << 16;
    const bool far_u = cu != rank, far_d = cd != rank;
    // a plain warp's edges all stay in this CTA: no test per store
    const bool plain_w = __all_sync(0xffffffffu, active && !far_u && !far_d && w == CX);
    unsigned flags = (active ? F_ACTIVE : 0u) | (h < RB ? F_SHORT : 0u) | (far_u ? F_FARU : 0u) | (far_d ? F_FARD : 0u) |
                     // warps holding a band whose neighbour is in another CTA wait for its rows
                     (__any_sync(0xffffffffu, far_u) ? F_NEEDU : 0u) | (__any_sync(0xffffffffu, far_d) ? F_NEEDD : 0u) |
                     (far_u && tc == 0 ? F_LEADU : 0u) | (far_d && tc == 0 ? F_LEADD : 0u) |   // one thread re-arms each mbarrier
                     // a warp holding the ragged right edge takes its ghost column (column 0's u) before its V phase
                     (__any_sync(0xffffffffu, w < CX) ? F_LATE : 0u) | (n_lo == 1 ? F_FIRST : 0u) |
                     (plain_w ? F_PLAIN : 0u) | (unsigned)(w - 1) << F_W | cu << F_CU | cd << F_CD;

    // projection of the sigma group: the threads holding measured cells stage their rows (two buffers by step
    // parity), after the next barrier thread e of the CTA moves the value of entry e to a history of two windows
    // of RES_WIN steps, and every RES_WIN steps the CTA forms s(n) = sum_e w_e F_e(n) of the window's steps,
    // one lane per step and group of entries (in FP64; GB300's FP64 pipe takes 64 clocks per warp
    // instruction, which a reduction per step put on the critical path of every step).
    // The terms w_n s(n) go to the second field buffer (unused otherwise), and rank 0 adds them at the end of
    // the launch as the multi-step kernels do: by tile and launch index (a CTA's entries of one tile are a
    // piece).  The sum over a run's steps is rounded to the last bit of its early terms thousands of times, the
    // force is a small difference of such sums, and in this order they round as before and do not depend on
    // how the steps were cut into launches.
    const DevResWarp pw = D.warps[(int)rank * (nt >> 5) + warp];
    unsigned pk_stage;             // first staged word (16 bits), element of this thread's entry (16 bits)
    const int stage_w = nt * SL::WORDS + D.gen_words, sbuf = D.stage_words;
    ResSums<R> sums{reinterpret_cast<double *>(dyn), reinterpret_cast<double *>(S.fields) + D.term_off, slot, piece, n_lo, S.tail_from + 1,
                    D.ctas[rank].np, D.ctas[rank].rounded};
    sums.layout(stage_w + 2 * sbuf, D);
    {
        flags |= ((pw.lanes >> lane) & 1) ? F_STAGE : 0u;
        flags |= pw.lanes ? F_STAGEW : 0u;
        flags |= pw.rows << F_ROWS;
        const int st = stage_w + pw.stage0 + __popc(pw.lanes & ((1u << lane) - 1u)) * pw.stride;
        for (int i = t; i < cnt; i += nt) sums.dd[sums.gw_i + i] = S.gw[n_lo - 1 + i];
        const DevResCta &pc = D.ctas[rank];
        int off = 0;
        for (int q = t; q < RES_PIECES * 32 + 1; q += nt) slot[q] = pc.slot[q];
        if (t < RES_PIECES) piece[t] = pc.piece[t];
        if (t < pc.ne) {
            flags |= F_MINE;
            off = D.ents[pc.e0 + t].off;
            sums.dd[sums.we_i + t] = D.ents[pc.e0 + t].w;
        }
        pk_stage = (unsigned)st | (unsigned)off << 16;
    }

    // the fields of the block with vx of the row above (vxm) and vy of the column to the left (vym), which
    // are updated here as well as by their owners so that one exchange of u per step is enough; and the
    // coefficients times their step factors (the first group's with hf, the sigma group's with bf, as in
    // step2d_tk.cu); the half step at n = 1 halves the first group
    R u[RB][CX], vx[RB][CX], vy[RB][CX], vxm[RED ? CX : 1], vym[RED ? RB : 1];   // vxm, vym with RED only
    const bool su = S.second_u != 0;
    R cxu, cyu, cuu;   // the coefficients of a warp whose cells are all of one material (those of vx negated, here and in the tables)
    const bool uni = pw.gen < 0;
    const V4 *const ow = blocks + nt * SL::WORDS + ((uni ? 0 : pw.gen) * 32 + lane) * SL::CWORDS;
    {
        const R *__restrict__ fu = reinterpret_cast<const R *>(S.fields);
        const R *__restrict__ fvx = fu + N;
        const R *__restrict__ fvy = fu + 2 * N;
        const R hf = (R)S.hf, bf = (R)S.bf;
        const R fV = (su ? hf : bf) * (su && n_lo == 1 ? (R)0.5 : (R)1), fU = (su ? bf : hf) * (!su && n_lo == 1 ? (R)0.5 : (R)1);
        const R *__restrict__ coef = reinterpret_cast<const R *>(S.coef);
        const uint8_t *__restrict__ mat = S.mat;
        V4 *const oc = const_cast<V4 *>(ow);
        R lf[KV * CX];
        const int xm = x0 == 0 ? nx - 1 : x0 - 1;
        auto grid_row = [&](int r) {   // of the cluster's row r
            const int y = r + D.shift;
            return y < 0 ? y + ny : (y >= ny ? y - ny : y);
        };
#pragma unroll
        for (int r = RED ? -1 : 0; r < RB; ++r) {
            V4 kx, ky, ku;
#pragma unroll
            for (int c = 0; c < CX; ++c) {
                R vu = (R)0, vvx = (R)0, vvy = (R)0;
                kx.c[c] = ky.c[c] = ku.c[c] = (R)0;
                if (active && r < h && c < w) {
                    const unsigned g = (unsigned)(grid_row(y0 + r) * nx + x0 + c);
                    vvx = fvx[g];
                    const int m = mat[g];
                    kx.c[c] = -fV * coef[3 * m + 1];
                    if (r >= 0) {
                        vu = fu[g];
                        vvy = fvy[g];
                        ku.c[c] = fU * coef[3 * m];
                        ky.c[c] = fV * coef[3 * m + 2];
                    }
                }
                if (r < 0) {
                    vxm[RED ? c : 0] = vvx;
                } else {
                    u[r < 0 ? 0 : r][c] = vu;
                    vx[r < 0 ? 0 : r][c] = vvx;
                    vy[r < 0 ? 0 : r][c] = vvy;
                }
            }
            if (!uni) {
                oc[SL::CVX + r + SL::RED] = kx;
                if (r >= 0) {
                    oc[SL::CVY + r] = ky;
                    oc[SL::CU + r] = ku;
                }
            }
            if (RED && r >= 0) {
                R v = (R)0, k = (R)0;
                if (active && r < h) {
                    const unsigned g = (unsigned)(grid_row(y0 + r) * nx + xm);
                    v = fvy[g];
                    k = fV * coef[3 * mat[g] + 2];
                }
                vym[RED && r >= 0 ? r : 0] = v;
                lf[r < 0 ? 0 : r] = k;
            }
        }
#pragma unroll
        for (int k = 0; k < KV; ++k) {
            V4 v;
#pragma unroll
            for (int c = 0; c < CX; ++c) v.c[c] = RED && k * CX + c < RB ? lf[k * CX + c] : (R)0;
            if (RED && !uni) oc[SL::CVYL + k] = v;
        }
        const unsigned act = __ballot_sync(0xffffffffu, active);
        int m0 = active ? mat[(unsigned)(grid_row(y0) * nx + x0)] : 0;
        m0 = __shfl_sync(0xffffffffu, m0, act ? __ffs(act) - 1 : 0);
        cuu = fU * coef[3 * m0];
        cxu = -fV * coef[3 * m0 + 1];
        cyu = fV * coef[3 * m0 + 2];
    }
    const R a = (R)S.a;
    if (multi) cluster_sync();   // every CTA of the cluster runs, its mbarriers initialised, before it is written to
    else __syncthreads();

    auto wait_far = [&](unsigned need, unsigned lead, unsigned mb, int i) {
        if (flags & need) {
            const unsigned m = mb + 8u * (i & 1);
            if (!mb_wait(m, ((unsigned)i >> 1) & 1u)) flags = (flags | F_DEAD) & ~F_EXCHANGE;
            if ((flags & lead) && i + 2 < cnt) mb_expect(m, D.tcols * 16);
        }
    };
    auto consume = [&](int i) {
        sums.consume(i, flags & F_MINE, reinterpret_cast<const R *>(blocks + stage_w + (i & 1) * sbuf), (int)(pk_stage >> 16));
    };
    auto put_row = [&](unsigned far, int at, unsigned cta, unsigned mb, const V4 &v) {
        if (flags & far) st_async(map_rank((unsigned)__cvta_generic_to_shared(blocks + at), cta), map_rank(mb, cta), v);
        else blocks[at] = v;
    };
    auto col_of = [&](const R (&f)[RB][CX], int c, int k) -> V4 {
        V4 v;
#pragma unroll
        for (int q = 0; q < CX; ++q) v.c[q] = k * CX + q < RB ? f[k * CX + q < RB ? k * CX + q : 0][c] : (R)0;
        return v;
    };
    auto last_row = [&](const R (&f)[RB][CX]) -> V4 {
        const bool cut = RB > 1 && (flags & F_SHORT);
        V4 v;
#pragma unroll
        for (int c = 0; c < CX; ++c) v.c[c] = cut ? f[RB > 1 ? RB - 2 : 0][c] : f[RB - 1][c];
        return v;
    };
    auto put_last_col = [&](const R (&f)[RB][CX], int at) {   // the last valid column, to the right
        if (flags & F_LATE) {
            const int w = (int)((flags >> F_W) & 3u) + 1;
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                R e = f[r][CX - 1];
#pragma unroll
                for (int c = 1; c < CX; ++c)
                    if (w == c) e = f[r][c - 1];
                reinterpret_cast<R *>(blocks + at)[r] = e;
            }
        } else {
#pragma unroll
            for (int k = 0; k < KV; ++k) blocks[at + k] = col_of(f, CX - 1, k);
        }
    };
    // the block's edges into the neighbours' slots (of buffer i & 1) for their phase of step i
    auto push_u = [&](int i) {
        const int o = RED ? (i & 1) * SL::BUF : 0;
        const int iu = (int)(pk_row & 0xffffu) + o, id = (int)(pk_row >> 16) + o, il = (int)(pk_col & 0xffffu) + o, ir = (int)(pk_col >> 16) + o;
        V4 top;
#pragma unroll
        for (int c = 0; c < CX; ++c) top.c[c] = u[0][c];
        if (flags & F_PLAIN) {
            blocks[iu] = top;
            if (RED) blocks[id] = last_row(u);
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                blocks[il + k] = col_of(u, 0, k);
                if (RED) blocks[ir + k] = col_of(u, CX - 1, k);
            }
        } else if (flags & F_ACTIVE) {
            put_row(F_FARU, iu, (flags >> F_CU) & 15u, mb_d + 8u * (i & 1), top);
            if (RED) put_row(F_FARD, id, flags >> F_CD, mb_u + 8u * (i & 1), last_row(u));
#pragma unroll
            for (int k = 0; k < KV; ++k) blocks[il + k] = col_of(u, 0, k);
            if (RED) put_last_col(u, ir);
        }
    };
    auto push_v = [&](int i) {   // without RED
        const int id = (int)(pk_row >> 16), ir = (int)(pk_col >> 16);
        if (flags & F_PLAIN) {
            blocks[id] = last_row(vx);
#pragma unroll
            for (int k = 0; k < KV; ++k) blocks[ir + k] = col_of(vy, CX - 1, k);
        } else if (flags & F_ACTIVE) {
            put_row(F_FARD, id, flags >> F_CD, mb_u + 8u * (i & 1), last_row(vx));
            put_last_col(vy, ir);
        }
    };

    auto march = [&](auto uni_tag, auto su_tag) {
        constexpr bool UNI = decltype(uni_tag)::value;
        constexpr bool SU = decltype(su_tag)::value;
        auto row = [&](int arr, int r) -> V4 {   // arr 0: vx (r from -1), 1: vy, 2: u
            if constexpr (UNI) {
                V4 v;
#pragma unroll
                for (int c = 0; c < CX; ++c) v.c[c] = arr == 0 ? cxu : (arr == 1 ? cyu : cuu);
                return v;
            } else {
                return ow[arr == 0 ? SL::CVX + r + SL::RED : (arr == 1 ? SL::CVY + r : SL::CU + r)];
            }
        };
        auto one = [&](int arr, int r, int c) -> R {
            if constexpr (UNI) return arr == 1 ? cyu : cuu;
            else return reinterpret_cast<const R *>(ow + (arr == 1 ? SL::CVY : SL::CU) + r)[c];
        };
        auto upx = [&](R v, R k, R d) -> R { return SU ? v + k * d : a * v + k * d; };   // k is negated
        auto upy = [&](R v, R k, R d) -> R { return SU ? v + k * d : a * v + k * d; };
        auto upu = [&](R v, R k, R d) -> R { return SU ? a * v + k * d : v + k * d; };
        // vx of a row from u of the row below it (`hi`) and its own (`lo`).  FP32 takes two cells per instruction,
        // with the operations and roundings of one at a time (x - y as y * -1 + x): 7.39 -> 7.15 us a step at
        // 128 x 128 (320 simulations), 757.8 -> 779.3 Gcell-updates/s on the 400 x 166 sweep.  u in pairs as well: 777.1,
        // and 0.747 -> 0.790 us a step on grids of a few warps (its differences along x are no aligned pairs).
        auto row_vx = [&](R (&f)[CX], const V4 &k, const R *hi, const R *lo) {
            if constexpr (sizeof(R) == 4) {
#pragma unroll
                for (int c = 0; c < CX; c += 2) {
                    const float2 v = make_float2(f[c], f[c + 1]), kk = make_float2(k.c[c], k.c[c + 1]);
                    const float2 d = __ffma2_rn(make_float2(lo[c], lo[c + 1]), make_float2(-1.0f, -1.0f), make_float2(hi[c], hi[c + 1]));
                    const float2 o = SU ? __ffma2_rn(kk, d, v) : __ffma2_rn(make_float2(a, a), v, __fmul2_rn(kk, d));
                    f[c] = o.x;
                    f[c + 1] = o.y;
                }
            } else {
#pragma unroll
                for (int c = 0; c < CX; ++c) f[c] = upx(f[c], k.c[c], hi[c] - lo[c]);
            }
        };
        auto stage = [&](int i) {
            if (flags & F_STAGE) {
                V4 *q = blocks + (pk_stage & 0xffffu) + (i & 1) * sbuf;
#pragma unroll
                for (int r = 0; r < RB; ++r)
                    if (flags & (1u << (F_ROWS + r))) {
                        V4 v;
                        if (SU) {
#pragma unroll
                            for (int c = 0; c < CX; ++c) v.c[c] = u[r][c];
                            *q++ = v;
                        } else {
#pragma unroll
                            for (int c = 0; c < CX; ++c) v.c[c] = vx[r][c];
                            *q++ = v;
#pragma unroll
                            for (int c = 0; c < CX; ++c) v.c[c] = vy[r][c];
                            *q++ = v;
                        }
                    }
            }
        };
        // u of row r: the cells whose u a neighbour needs, and the others
        auto row_u = [&](int r, bool edge, bool inner) {
            const V4 k = row(2, r);
#pragma unroll
            for (int c = 0; c < CX; ++c) {
                const bool is_edge = r == 0 || r + 2 >= RB || c == 0 || c == CX - 1;
                if (is_edge ? edge : inner)
                    u[r][c] = upu(u[r][c], k.c[c], (vy[r][c] - (c > 0 ? vy[r][c > 0 ? c - 1 : 0] : vym[RED ? r : 0])) - (vx[r][c] - (r > 0 ? vx[r > 0 ? r - 1 : 0][c] : vxm[RED ? c : 0])));
            }
        };
        [[maybe_unused]] constexpr bool HAS_INNER = RB > 3 && CX > 2;   // cells whose u no neighbour needs
        // RED: vx of the row above from its u
        auto v_up = [&](const V4 *own) {
            if constexpr (RED) {
                const V4 hu = own[SL::UP], k = row(0, -1);
                row_vx(vxm, k, u[0], hu.c);
            }
        };
        // vx of the last rows from u of the row below
        auto v_down = [&](const V4 *own) {
            const V4 hd = own[SL::DN];
            if (RB > 1) {
                // a band of RB - 1 rows keeps its neighbour's row 0 in its last row
                const bool cut = flags & F_SHORT;
#pragma unroll
                for (int c = 0; c < CX; ++c) u[RB - 1][c] = cut ? hd.c[c] : u[RB - 1][c];
                const V4 k = row(0, RB > 1 ? RB - 2 : 0);
                row_vx(vx[RB > 1 ? RB - 2 : 0], k, u[RB - 1], u[RB > 1 ? RB - 2 : 0]);
            }
            const V4 k = row(0, RB - 1);
            row_vx(vx[RB - 1], k, hd.c, u[RB - 1]);
        };
        // V phase: the part no neighbour's u enters, the step's barrier, the columns at the sides (RED), the rest
        auto phase_v = [&](int i) {
            const V4 *const own = blocks + (int)threadIdx.x * SL::WORDS + (RED ? (i & 1) * SL::BUF : 0);
            if (flags & F_LATE) {
                __syncthreads();
                const R *const hr = reinterpret_cast<const R *>(own + SL::RT);
                const int w = (int)((flags >> F_W) & 3u) + 1;
#pragma unroll
                for (int r = 0; r < RB; ++r)
#pragma unroll
                    for (int c = 1; c < CX; ++c)
                        if (w == c) u[r][c] = hr[r];
            }
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                if (CX > 1) {
                    const V4 k = row(1, r);
#pragma unroll
                    for (int c = 0; c + 1 < CX; ++c) vy[r][c] = upy(vy[r][c], k.c[c], u[r][c + 1] - u[r][c]);
                }
                if (r + 2 < RB) {
                    const V4 k = row(0, r);
                    row_vx(vx[r], k, u[r + 1], u[r]);
                }
            }
            if (!(flags & F_LATE)) __syncthreads();
            if ((RED || SU) && i > 0) consume(i - 1);
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                const V4 hr = own[SL::RT + k];
                [[maybe_unused]] V4 hl, kl;
                if constexpr (RED) {
                    hl = own[SL::LF + k];
                    if constexpr (UNI) {
#pragma unroll
                        for (int c = 0; c < CX; ++c) kl.c[c] = cyu;
                    } else {
                        kl = ow[SL::CVYL + k];
                    }
                }
#pragma unroll
                for (int c = 0; c < CX; ++c)
                    if (k * CX + c < RB) {
                        const int r = k * CX + c < RB ? k * CX + c : 0;
                        if constexpr (RED) vym[RED ? r : 0] = upy(vym[RED ? r : 0], kl.c[c], u[r][0] - hl.c[c]);
                        vy[r][CX - 1] = upy(vy[r][CX - 1], one(1, r, CX - 1), hr.c[c] - u[r][CX - 1]);
                    }
            }
            if constexpr (!RED) {
                wait_far(F_NEEDD, F_LEADD, mb_d, i);
                v_down(own);
            }
        };
        // U phase without RED: the part no neighbour's v enters, the barrier, the rest
        auto phase_u = [&](int i) {
            const V4 *const own = blocks + (int)threadIdx.x * SL::WORDS;
#pragma unroll
            for (int r = 1; r < RB; ++r) {
                const V4 k = row(2, r);
#pragma unroll
                for (int c = 1; c < CX; ++c) u[r][c] = upu(u[r][c], k.c[c], (vy[r][c] - vy[r][c - 1]) - (vx[r][c] - vx[r - 1][c]));
            }
            __syncthreads();
            if (!SU && i > 0) consume(i - 1);
            R hl0 = (R)0;
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                const V4 hl = own[SL::LF + k];
                if (k == 0) hl0 = hl.c[0];
#pragma unroll
                for (int c = 0; c < CX; ++c)
                    if (k * CX + c < RB && k * CX + c > 0) {
                        const int r = k * CX + c < RB && k * CX + c > 0 ? k * CX + c : 1;
                        u[r < RB ? r : 0][0] = upu(u[r < RB ? r : 0][0], one(2, r, 0), (vy[r < RB ? r : 0][0] - hl.c[c]) - (vx[r < RB ? r : 0][0] - vx[r < RB ? r - 1 : 0][0]));
                    }
            }
            wait_far(F_NEEDU, F_LEADU, mb_u, i);
            const V4 hv = own[SL::UP], k = row(2, 0);
#pragma unroll
            for (int c = 0; c < CX; ++c)
                u[0][c] = upu(u[0][c], k.c[c], (vy[0][c] - (c > 0 ? vy[0][c > 0 ? c - 1 : 0] : hl0)) - (vx[0][c] - hv.c[c]));
        };
        auto full_scale = [&] {   // after the half step: the first group's coefficients take their full value
            if (flags & F_FIRST) {
                flags &= ~F_FIRST;
                if constexpr (UNI) {
                    if (SU) {
                        cxu *= (R)2;
                        cyu *= (R)2;
                    } else {
                        cuu *= (R)2;
                    }
                } else {
                    R *const o = reinterpret_cast<R *>(const_cast<V4 *>(ow));
#pragma unroll 1
                    for (int q = SU ? SL::CVX * CX : SL::CU * CX; q < (SU ? SL::CU * CX : (SL::CU + RB) * CX); ++q) o[q] *= (R)2;
                }
            }
        };

        if constexpr (RED) {
            if (!SU) {
#pragma unroll
                for (int r = 0; r < RB; ++r) row_u(r, true, true);
                full_scale();
            }
            push_u(0);
        } else {
            if (SU) push_u(0);
            else push_v(0);
        }
#pragma unroll 1
        for (int i = 0; i < cnt; ++i) {
            // opaque to the compiler, which would otherwise keep every unpacked value live through the loop
            asm volatile("" : "+r"(flags), "+r"(pk_row), "+r"(pk_col), "+r"(pk_stage));
            if constexpr (RED) {
                phase_v(i);
                const V4 *const own = blocks + (int)threadIdx.x * SL::WORDS + (i & 1) * SL::BUF;
                wait_far(F_NEEDU, F_LEADU, mb_u, i);
                v_up(own);
                wait_far(F_NEEDD, F_LEADD, mb_d, i);
                v_down(own);
                if (!SU) stage(i);
                if (SU || i + 1 < cnt) {
#pragma unroll
                    for (int r = 0; r < RB; ++r) row_u(r, true, false);
                    if (flags & (SU ? F_STAGEW | F_LATE : F_LATE)) {   // staged cells, and a ragged last column, are ready before the step's barrier
#pragma unroll
                        for (int r = 0; r < RB; ++r)
                            if (HAS_INNER) row_u(r, false, true);
                        if (SU) stage(i);
                        if (i + 1 < cnt) push_u(i + 1);
                    } else {
                        if (i + 1 < cnt) push_u(i + 1);
#pragma unroll
                        for (int r = 0; r < RB; ++r)
                            if (HAS_INNER) row_u(r, false, true);
                    }
                }
                if (SU) full_scale();
            } else {
                if (SU) {
                    phase_v(i);
                    push_v(i);
                    phase_u(i);
                    stage(i);
                    if (i + 1 < cnt) push_u(i + 1);
                } else {
                    phase_u(i);
                    push_u(i);
                    phase_v(i);
                    stage(i);
                    if (i + 1 < cnt) push_v(i + 1);
                }
                full_scale();
            }
        }
        __syncthreads();
        consume(cnt - 1);
    };
    if (su) {
        if (uni) march(ResFlag<true>{}, ResFlag<true>{});
        else march(ResFlag<false>{}, ResFlag<true>{});
    } else {
        if (uni) march(ResFlag<true>{}, ResFlag<false>{});
        else march(ResFlag<false>{}, ResFlag<false>{});
    }

    // where the block lies, worked out again (kept through the loop it would cost it registers)
    int t2 = threadIdx.x;
    asm volatile("" : "+r"(t2));
    const bool dead = flags & F_DEAD;
    {
        const int lb = t2 / D.tcols, tc = t2 - lb * D.tcols, b = (int)cluster_rank() * D.nb / (int)cluster_size() + lb;
        const int y0 = b * S.ny / D.nb, x0 = tc * CX, h = (flags & F_SHORT) ? RB - 1 : RB, w = (int)((flags >> F_W) & 3u) + 1;
        const unsigned N = (unsigned)S.nx * (unsigned)S.ny;
        R *const f = reinterpret_cast<R *>(S.fields);
        if (flags & F_ACTIVE) {
#pragma unroll
            for (int r = 0; r < RB; ++r)
#pragma unroll
                for (int c = 0; c < CX; ++c)
                    if (r < h && c < w) {
                        const int y = y0 + r + D.shift;
                        const unsigned g = (unsigned)((y >= S.ny ? y - S.ny : y) * S.nx + x0 + c);
                        f[g] = u[r][c];
                        f[N + g] = vx[r][c];
                        f[2 * N + g] = vy[r][c];
                    }
        }
    }
    if (dead) *D.status = 1;
    sums.finish(D, cnt, S.acc, S.tail);
    if (dead) linger();
}

}  // namespace

template <typename R, int RB>
static const void *res2d_fn() { return (const void *)k_res2d<R, RB, RES_MAXT>; }

static const void *res_kernel(int cyl, int fp64, int rb)
{
    if (cyl) return rescyl_kernel(fp64, rb);
    if (fp64) return rb == 1 ? res2d_fn<double, 1>() : rb == 2 ? res2d_fn<double, 2>() : rb == 4 ? res2d_fn<double, 4>() : nullptr;
    return rb == 2 ? res2d_fn<float, 2>() : rb == 4 ? res2d_fn<float, 4>() : nullptr;
}

int res_words(int cyl, int fp64, int rb, int *coef)   // Slots<R, rb>::WORDS, CWORDS
{
    if (cyl) return rescyl_words(fp64, rb, coef);
    const int cx = fp64 ? 2 : 4, kv = (rb + cx - 1) / cx, red = fp64 ? 0 : 1;
    *coef = (3 * rb + red * (1 + kv)) | 1;
    return ((1 + red) * (2 + 2 * kv)) | 1;
}

int res2d_proj_bytes(const Res2dShape &q)
{
    const int rs = q.fp64 ? 8 : 4;
    return (q.ne_max + q.np_max * 16 * RES_WIN + 2 * q.ntile_max * RES_LAUNCH_INDICES) * 8 +
           (2 * RES_WIN * q.ne_max * rs + 15) / 16 * 16;
}

cudaError_t res2d_prepare()
{
    for (int f = 0; f < 4; ++f)
        for (int rb : {1, 2, 3, 4}) {
            const void *k = res_kernel(f >> 1, f & 1, rb);
            if (!k) continue;
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, RES_SMEM_MAX);
            if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
            if (e != cudaSuccess) return e;
        }
    return cudaSuccess;
}

static cudaError_t launch_cfg(const void *k, int grid, int cluster, int threads, int smem, cudaStream_t st, cudaLaunchConfig_t *cfg,
                              cudaLaunchAttribute *at)
{
    *cfg = cudaLaunchConfig_t{};
    cfg->gridDim = dim3((unsigned)grid);
    cfg->blockDim = dim3((unsigned)threads);
    cfg->dynamicSmemBytes = (size_t)smem;
    cfg->stream = st;
    at->id = cudaLaunchAttributeClusterDimension;
    at->val.clusterDim.x = (unsigned)cluster;
    at->val.clusterDim.y = 1;
    at->val.clusterDim.z = 1;
    cfg->attrs = at;
    cfg->numAttrs = 1;
    return k ? cudaSuccess : cudaErrorInvalidValue;
}

void launch_res2d(const Res2dShape &q, const void *sims, int nsims, int64_t launch, int count, cudaStream_t st)
{
    if (nsims <= 0) return;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    const void *k = res_kernel(q.cyl, q.fp64, q.rb);
    if (launch_cfg(k, nsims * q.cluster, q.cluster, q.threads, q.smem, st, &cfg, &at) != cudaSuccess) return;
    void *args[] = {(void *)&sims, (void *)&launch, (void *)&count};
    cudaLaunchKernelExC(&cfg, k, args);
}

// Clusters of `q`'s size resident at once: with one CTA per SM (`alone`), or as many as fit.
static int clusters_resident(const void *k, const Res2dShape &q, bool alone)
{
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at;
    launch_cfg(k, q.cluster, q.cluster, q.threads, alone ? RES_SMEM_MAX : q.smem, nullptr, &cfg, &at);
    int fit = 0;
    if (cudaOccupancyMaxActiveClusters(&fit, k, &cfg) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return fit;
}

// The model's clocks of a step, `share` CTAs to an SM, for the warps that share it: FP32 the larger of 137 a warp (measured with 16 warps; about 300
// instructions a warp, 45% of the issue slots) and of one warp's own chain (1200; 1750 when rows come from other CTAs);
// FP64 its arithmetic at two lanes a clock and SM times 1.22, plus 700.  Simulations beyond those resident
// at once run one after the other.  Measured in FP32 (Gcell-updates/s, 400 x 166 cells, 640 simulations,
// without the projection, which costs 13%): 4 rows in clusters of 9: 870, of 10: 749; 6 and 7 rows: 700 at
// most (fewer threads fit the shared memory); the three-step kernel 465 with its projection.  Grids larger
// than a cluster of 16 holds stay with that kernel, at 539 on 512 x 512 (256 simulations).  Every shape that
// fits is taken: against the multi-step kernels the worst, clusters of 11 to 14 that leave a third of the SMs
// idle, ran at 436 : 409 (FP32, 400 x 200, 320 simulations) and 30.1 : 28.5 (FP64, 256 x 200, 160).  Cylindrical, FP32: 27.5 clocks a
// warp and cell of a thread (29 with three rows, which spill a little) and 770, at least 2300; 126 simulations of
// 60 x 400: two rows in clusters of 6 229 Gcell-updates/s, of 7 177, of 9 202, three rows in clusters of 5 220, of 6 224.
static double step_clocks(const Res2dShape &q, int share)
{
    const int cx = q.fp64 ? 2 : 4;
    const double warps = share * (q.threads / 32);
    if (q.cyl) return q.fp64 ? 1.22 * warps * 16.0 * q.rb * cx * 40.0 + 1000.0 : std::max(2300.0, warps * q.rb * cx * (q.rb == 3 ? 29.0 : 27.5) + 770.0);
    if (q.fp64) return 1.22 * warps * 16.0 * q.rb * cx * 9.0 + 700.0;
    const double chain = q.cluster > 1 ? 1750.0 : 1200.0, issue = (q.rb == 4 ? 137.0 : 120.0) * warps;
    return std::max(chain, issue) + 0.1 * std::min(chain, issue);
}

static bool later(double t, int order, double t2, int order2) { return t != t2 ? t > t2 : order > order2; }

ResShapes::ResShapes(int cyl, int fp64, int nx, int ny, int nsims_) : nsims(nsims_)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return;
    }
    const int cx = fp64 ? 2 : 4;
    const int tcols = (nx + cx - 1) / cx;
    for (int rb : {1, 2, 3, 4}) {
        if (!res_kernel(cyl, fp64, rb)) continue;
        const int nb = (ny + rb - 1) / rb;                       // bands of rb or rb - 1 rows
        if (rb > 1 && ny / nb < rb - 1) continue;
        for (int c = 1; c <= RES_CLUSTER_MAX && c <= nb; ++c) {
            const int bpc = (nb + c - 1) / c, threads = (tcols * bpc + 31) / 32 * 32;
            if (threads > RES_MAXT) continue;
            Res2dShape q{};
            q.fp64 = fp64;
            q.cyl = cyl;
            q.rb = rb;
            q.cluster = c;
            q.threads = threads;
            q.tcols = tcols;
            q.nb = nb;
            int cw = 0;
            q.smem = (threads * res_words(cyl, fp64, rb, &cw) + (cyl ? RES_RAD * tcols : 0)) * 16 + RES_LAUNCH_STEPS * 8;   // (cyl: radial factors)
            if (q.smem > RES_SMEM_MAX) continue;
            // With `share` CTAs to an SM no more clusters run at once than the SMs hold so many times, nor than the
            // SMs' shared memory (228 KB, 1 KB of it a CTA's own) and threads allow.
            const int alone = std::max(1, sms / c);
            const int most = std::max(alone, sms * std::min(228 * 1024 / (q.smem + 1024), 2048 / threads) / c);
            double t = 0;
            for (int share = 1; share == 1 || (share - 1) * alone < std::min(most, nsims); ++share) {
                const int at_once = std::min(most, alone * share);
                const double ts = (nsims + at_once - 1) / at_once * step_clocks(q, share);
                if (share == 1 || ts < t) t = ts;
            }
            heap.push_back({t, (int)heap.size(), false, q});
        }
    }
    std::make_heap(heap.begin(), heap.end(), [](const Shape &x, const Shape &y) { return later(x.t, x.order, y.t, y.order); });
}

bool ResShapes::next(Res2dShape *q, double *clocks)
{
    const auto cmp = [](const Shape &x, const Shape &y) { return later(x.t, x.order, y.t, y.order); };
    while (!heap.empty()) {
        std::pop_heap(heap.begin(), heap.end(), cmp);
        Shape &s = heap.back();
        if (s.exact) {
            *q = s.q;
            if (clocks) *clocks = s.t;
            heap.pop_back();
            return true;
        }
        const void *k = res_kernel(s.q.cyl, s.q.fp64, s.q.rb);
        const int fit1 = clusters_resident(k, s.q, true);
        // CTAs on an SM: one if each simulation's cluster finds SMs of its own
        const int fit = nsims > fit1 ? std::max(fit1, clusters_resident(k, s.q, false)) : fit1;
        if (fit1 < 1) {
            heap.pop_back();
            continue;
        }
        const int share = std::max(1, std::min((nsims + fit1 - 1) / fit1, fit / fit1));
        const int waves = (nsims + fit1 * share - 1) / (fit1 * share);
        s.t = waves * step_clocks(s.q, share);
        s.exact = true;
        std::push_heap(heap.begin(), heap.end(), cmp);
    }
    return false;
}

}  // namespace cas
