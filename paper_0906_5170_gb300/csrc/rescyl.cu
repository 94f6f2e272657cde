// Resident march of the cylindrical (r, z) cross-sections (Sec. III C: fields ~ exp(i m phi) in the
// real-phase form): a thread-block cluster holds one simulation's six fields in registers and advances it
// through a whole chunk of time steps per launch, as res2d.cu does for the TM/TE simulations.
//
// The update is that of step6m.cu's and step6c2.cu's cylindrical marches, value for value: curls with
// d/dphi -> +-m, r-weighted radial differences, the Stokes form on the axis; the first group's step is a
// half step at n = 1.  A thread owns CX columns (16 bytes, along r) by RB rows (along z).  Per step
//   H from E of the cell, E_r and E_phi of the row below, E_z and E_phi of the column to the right
//   E from H of the cell, H_r and H_phi of the row above, H_z and H_phi of the column to the left
// (electric sources H then E, magnetic ones E then H).  After a group's update its edges go to the
// neighbours' slots; the cells that need no neighbour come before the phase's barrier, the others after it.
//
// Bound by the latency of one warp's chain and its two barriers a step rather than by memory: 126
// simulations of 60 x 400 cells run at 229 Gcell-updates/s in FP32 (72 with two steps per launch through
// memory; 115 while the radial factors' loads met in the same banks), in FP64 at 13.4 (4.5).
#include "resident.cuh"

namespace cas {

namespace {

// 16-byte words of a thread's slots: rows E_r, E_phi from below and H_r, H_phi from above, columns E_z,
// E_phi from the right and H_z, H_phi from the left; and of its coefficients (E_r .. H_phi rows)
template <typename R, int RB>
struct SlotsC {
    static constexpr int CX = 16 / (int)sizeof(R);
    static constexpr int KV = (RB + CX - 1) / CX;
    static constexpr int ED = 0, HU = 2, ER = 4, HL = 4 + 2 * KV;
    static constexpr int WORDS = (4 + 4 * KV) | 1;
    static constexpr int CWORDS = (6 * RB) | 1;
};

template <typename R, int RB, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
k_rescyl(const DevResCyl *__restrict__ sims, int64_t launch, int count)
{
    using V4 = Vec16<R>;
    using SL = SlotsC<R, RB>;
    constexpr int CX = SL::CX, KV = SL::KV;
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ short slot[RES_PIECES * 32 + 1];
    __shared__ short piece[RES_PIECES];
    __shared__ __align__(8) unsigned long long mbar[4];   // rows from the previous and from the next CTA, by step parity

    const unsigned C = cluster_size(), rank = cluster_rank();
    const DevResCyl &D = sims[blockIdx.x / C];
    const DevSim6 &S = D.s;
    const int64_t L0 = launch - S.s0;
    const int64_t l_lo = L0 > 1 ? L0 : 1, l_hi = L0 + count - 1;
    if (l_hi < l_lo || (l_lo - 1) * D.k + 1 > S.T) return;
    const int n_lo = (int)((l_lo - 1) * D.k + 1), n_hi = (int)min((int64_t)S.T, l_hi * D.k);
    const int cnt = n_hi - n_lo + 1;
    const bool multi = C > 1;

    const int nt = blockDim.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int nx = S.n[0], ny = S.n[1], nb = D.nb, tcols = D.tcols;
    const unsigned N = (unsigned)nx * (unsigned)ny;
    const int b0 = (int)rank * nb / (int)C, b1 = ((int)rank + 1) * nb / (int)C;
    const int lb = t / tcols, tc = t - lb * tcols, b = b0 + lb;
    const bool active = b < b1;
    const int y0 = active ? b * ny / nb : 0;
    const int h = active ? (b + 1) * ny / nb - y0 : RB;
    const int x0 = tc * CX;
    const int w = active ? min(CX, nx - x0) : CX;

    const unsigned mb_u = (unsigned)__cvta_generic_to_shared(&mbar[0]), mb_d = mb_u + 16;
    if (multi && t == 0) {
        for (int q = 0; q < 4; ++q) mb_init(mb_u + 8 * q, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        for (int q = 0; q < 4; ++q) mb_expect(mb_u + 8 * q, 2 * tcols * 16);   // two rows
    }

    V4 *const blocks = reinterpret_cast<V4 *>(dyn);
    const int own_i = t * SL::WORDS;
    const V4 *const own = blocks + own_i;
    unsigned cu = rank, cd = rank;   // the CTAs of the bands above and below
    auto band_slot = [&](int bb, unsigned *cta) {
        unsigned r = rank;
        if (bb < b0 || bb >= b1)
            r = (bb == (b1 == nb ? 0 : b1)) ? (rank + 1 == C ? 0 : rank + 1) : (rank == 0 ? C - 1 : rank - 1);
        *cta = r;
        return ((bb - (int)r * nb / (int)C) * tcols + tc) * SL::WORDS;
    };
    const int iu = (active ? band_slot(b == 0 ? nb - 1 : b - 1, &cu) : own_i) + SL::ED;
    const int id = (active ? band_slot(b + 1 == nb ? 0 : b + 1, &cd) : own_i) + SL::HU;
    const int il = own_i + (tc == 0 ? tcols - 1 : -1) * SL::WORDS + SL::ER;
    const int ir = own_i + (tc == tcols - 1 ? 1 - tcols : 1) * SL::WORDS + SL::HL;
    unsigned pk_row = (unsigned)iu | (unsigned)id << 16, pk_col = (unsigned)(active ? il : own_i) | (unsigned)(active ? ir : own_i) << 16;
    const bool far_u = cu != rank, far_d = cd != rank;
    const bool plain_w = __all_sync(0xffffffffu, active && !far_u && !far_d && w == CX);
    unsigned flags = (active ? F_ACTIVE : 0u) | (h < RB ? F_SHORT : 0u) | (far_u ? F_FARU : 0u) | (far_d ? F_FARD : 0u) |
                     (__any_sync(0xffffffffu, far_u) ? F_NEEDU : 0u) | (__any_sync(0xffffffffu, far_d) ? F_NEEDD : 0u) |
                     (far_u && tc == 0 ? F_LEADU : 0u) | (far_d && tc == 0 ? F_LEADD : 0u) |
                     (__any_sync(0xffffffffu, w < CX) ? F_LATE : 0u) | (n_lo == 1 ? F_FIRST : 0u) |
                     (plain_w ? F_PLAIN : 0u) | (unsigned)(w - 1) << F_W | cu << F_CU | cd << F_CD;

    // projection of the sigma group, as in res2d.cu (three components a staged row)
    const DevResWarp pw = D.warps[(int)rank * (nt >> 5) + warp];
    unsigned pk_stage;
    const int stage_w = nt * SL::WORDS + D.gen_words + RES_RAD * tcols, sbuf = D.stage_words;
    ResSums<R> sums{reinterpret_cast<double *>(dyn), reinterpret_cast<double *>(S.fields) + D.term_off, slot, piece, n_lo, S.tail_from + 1,
                    D.ctas[rank].np, D.ctas[rank].rounded};
    sums.layout(stage_w + 2 * sbuf, D);
    {
        flags |= ((pw.lanes >> lane) & 1) ? F_STAGE : 0u;
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

    // radial factors of the CTA's columns (step6c2.cu's, with kA or kB where they enter): 8 rows of CX per thread
    // column, RES_RAD words apart (8 apart, all lanes of a load met in the same banks)
    const R bxr = (R)S.bre[0], idx = (R)S.inv_dx;
    V4 *const rad = blocks + nt * SL::WORDS + D.gen_words;
    for (int q = t; q < tcols; q += nt) {
        const R kA = (R)S.kzA, kB = (R)S.kzB, ix = (R)S.inv_dx;
        V4 f[8];
#pragma unroll
        for (int c = 0; c < CX; ++c) {
            const int col = q * CX + c;
            const R ci = (R)col, ch = ci + (R)0.5;
            const R inv_ri = col > 0 ? ix / ci : (R)0, inv_rh = ix / ch;
            f[0].c[c] = kA * inv_ri;
            f[1].c[c] = kA * inv_rh;
            f[2].c[c] = (ci + (R)1) / ch;                                // ga
            f[3].c[c] = ci / ch;                                         // gb
            f[4].c[c] = kB * inv_rh;
            f[5].c[c] = kB * inv_ri;
            f[6].c[c] = col > 0 ? ch / ci : (R)4;                        // fa
            f[7].c[c] = col > 0 ? (ci - (R)0.5) / ci : (R)0;             // fb
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) rad[q * RES_RAD + k] = f[k];
    }
    const V4 *const my_rad = rad + tc * RES_RAD;

    R e[3][RB][CX], hh[3][RB][CX];
    const bool electric = S.magnetic == 0;
    R kE[3], kH[3];   // the coefficients of a warp whose cells are all of one material, times the group's step
    const bool uni = pw.gen < 0;
    const V4 *const ow = blocks + nt * SL::WORDS + ((uni ? 0 : pw.gen) * 32 + lane) * SL::CWORDS;
    {
        const R *__restrict__ f = reinterpret_cast<const R *>(S.fields);
        const R first = (R)(n_lo == 1 ? 0.5 * S.dt : S.dt), bs = (R)S.bs;
        const R bE = electric ? bs : first, bH = electric ? first : bs;
        const R *__restrict__ coef = reinterpret_cast<const R *>(S.coef);
        const uint8_t *__restrict__ mat = S.mat;
        V4 *const oc = const_cast<V4 *>(ow);
        auto grid_row = [&](int r) {
            const int y = r + D.shift;
            return y >= ny ? y - ny : y;
        };
#pragma unroll
        for (int r = 0; r < RB; ++r) {
            V4 k6[6];
#pragma unroll
            for (int c = 0; c < CX; ++c) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    e[k][r][c] = hh[k][r][c] = (R)0;
                    k6[k].c[c] = k6[3 + k].c[c] = (R)0;
                }
                if (active && r < h && c < w) {
                    const unsigned g = (unsigned)(grid_row(y0 + r) * nx + x0 + c);
                    const R *cm = coef + 6 * mat[g];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        e[k][r][c] = f[(unsigned)k * N + g];
                        hh[k][r][c] = f[(unsigned)(3 + k) * N + g];
                        k6[k].c[c] = bE * cm[k];
                        k6[3 + k].c[c] = bH * cm[3 + k];
                    }
                }
            }
            if (!uni) {
#pragma unroll
                for (int k = 0; k < 6; ++k) oc[k * RB + r] = k6[k];
            }
        }
        const unsigned act = __ballot_sync(0xffffffffu, active);
        int m0 = active ? mat[(unsigned)(grid_row(y0) * nx + x0)] : 0;
        m0 = __shfl_sync(0xffffffffu, m0, act ? __ffs(act) - 1 : 0);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            kE[k] = bE * coef[6 * m0 + k];
            kH[k] = bH * coef[6 * m0 + 3 + k];
        }
    }
    const R a = (R)S.a;
    const R xl = tc == 0 ? bxr : (R)1, xr = active && x0 + CX >= nx ? bxr : (R)1;   // factor of the columns across the axis and the wall
    if (multi) cluster_sync();
    else __syncthreads();

    auto wait_far = [&](unsigned need, unsigned lead, unsigned mb, int i) {
        if (flags & need) {
            const unsigned m = mb + 8u * (i & 1);
            if (!mb_wait(m, ((unsigned)i >> 1) & 1u)) flags = (flags | F_DEAD) & ~F_EXCHANGE;
            if ((flags & lead) && i + 2 < cnt) mb_expect(m, 2 * D.tcols * 16);
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
    auto put_last_col = [&](const R (&f)[RB][CX], int at) {
        if (flags & F_LATE) {
            const int w = (int)((flags >> F_W) & 3u) + 1;
#pragma unroll
            for (int r = 0; r < RB; ++r) {
                R v = f[r][CX - 1];
#pragma unroll
                for (int c = 1; c < CX; ++c)
                    if (w == c) v = f[r][c - 1];
                reinterpret_cast<R *>(blocks + at)[r] = v;
            }
        } else {
#pragma unroll
            for (int k = 0; k < KV; ++k) blocks[at + k] = col_of(f, CX - 1, k);
        }
    };
    // E_r and E_phi of row 0 to the band above, E_z and E_phi of column 0 to the left
    auto push_e = [&](int i) {
        const int iu = (int)(pk_row & 0xffffu), il = (int)(pk_col & 0xffffu);
        V4 r0, r2;
#pragma unroll
        for (int c = 0; c < CX; ++c) {
            r0.c[c] = e[0][0][c];
            r2.c[c] = e[2][0][c];
        }
        if (flags & F_PLAIN) {
            blocks[iu] = r0;
            blocks[iu + 1] = r2;
        } else if (flags & F_ACTIVE) {
            const unsigned cta = (flags >> F_CU) & 15u;
            put_row(F_FARU, iu, cta, mb_d + 8u * (i & 1), r0);
            put_row(F_FARU, iu + 1, cta, mb_d + 8u * (i & 1), r2);
        }
        if (flags & F_ACTIVE) {
#pragma unroll
            for (int k = 0; k < KV; ++k) {
                blocks[il + k] = col_of(e[1], 0, k);
                blocks[il + KV + k] = col_of(e[2], 0, k);
            }
        }
    };
    // H_r and H_phi of the last row to the band below, H_z and H_phi of the last column to the right
    auto push_h = [&](int i) {
        const int id = (int)(pk_row >> 16), ir = (int)(pk_col >> 16);
        if (flags & F_PLAIN) {
            blocks[id] = last_row(hh[0]);
            blocks[id + 1] = last_row(hh[2]);
        } else if (flags & F_ACTIVE) {
            const unsigned cta = flags >> F_CD;
            put_row(F_FARD, id, cta, mb_u + 8u * (i & 1), last_row(hh[0]));
            put_row(F_FARD, id + 1, cta, mb_u + 8u * (i & 1), last_row(hh[2]));
        }
        if (flags & F_ACTIVE) {
            put_last_col(hh[1], ir);
            put_last_col(hh[2], ir + KV);
        }
    };

    auto march = [&](auto uni_tag, auto el_tag) {
        constexpr bool UNI = decltype(uni_tag)::value;
        constexpr bool EL = decltype(el_tag)::value;
        auto row = [&](int k, int r) -> V4 {   // coefficient k (E_r .. H_phi) of row r
            if constexpr (UNI) {
                V4 v;
#pragma unroll
                for (int c = 0; c < CX; ++c) v.c[c] = k < 3 ? kE[k < 3 ? k : 0] : kH[k < 3 ? 0 : k - 3];
                return v;
            } else {
                return ow[k * RB + r];
            }
        };
        const R aH = EL ? (R)1 : a, aE = EL ? a : (R)1;
        // H of cell (r, c) from E_r, E_phi of the row below and E_z, E_phi of the column to the right
        auto cell_h = [&](int r, int c, R e0n, R e2n, R e1r, R e2r, const V4 &q0, const V4 &q1, const V4 &q2, const V4 &fri, const V4 &frh, const V4 &ga,
                          const V4 &gb) {
            const R dyEz = (e2n - e[2][r][c]) * idx, dyEx = (e0n - e[0][r][c]) * idx;
            const R dxEy = (e1r - e[1][r][c]) * idx;
            const R dxEphi = (e2r * ga.c[c] - e[2][r][c] * gb.c[c]) * idx;
            hh[0][r][c] = hh[0][r][c] * aH - (e[1][r][c] * fri.c[c] - dyEz) * q0.c[c];
            hh[1][r][c] = hh[1][r][c] * aH - (dxEphi - e[0][r][c] * frh.c[c]) * q1.c[c];
            hh[2][r][c] = hh[2][r][c] * aH - (dyEx - dxEy) * q2.c[c];
        };
        auto cell_e = [&](int r, int c, R h0p, R h2p, R h1l, R h2l, const V4 &q0, const V4 &q1, const V4 &q2, const V4 &frh, const V4 &fri, const V4 &fa,
                          const V4 &fb) {
            const R dyHz = (hh[2][r][c] - h2p) * idx, dyHx = (hh[0][r][c] - h0p) * idx;
            const R dxHy = (hh[1][r][c] - h1l) * idx;
            const R dxHphi = (hh[2][r][c] * fa.c[c] - h2l * fb.c[c]) * idx;
            const R c0 = hh[1][r][c] * frh.c[c] - dyHz;
            const R c1 = dxHphi - hh[0][r][c] * fri.c[c];
            const R c2 = dyHx - dxHy;
            e[0][r][c] = e[0][r][c] * aE + c0 * q0.c[c];
            e[1][r][c] = e[1][r][c] * aE + c1 * q1.c[c];
            e[2][r][c] = e[2][r][c] * aE + c2 * q2.c[c];
        };
        auto stage = [&](int i) {
            if (flags & F_STAGE) {
                V4 *q = blocks + (pk_stage & 0xffffu) + (i & 1) * sbuf;
#pragma unroll
                for (int r = 0; r < RB; ++r)
                    if (flags & (1u << (F_ROWS + r))) {
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            V4 v;
#pragma unroll
                            for (int c = 0; c < CX; ++c) v.c[c] = EL ? e[k][r][c] : hh[k][r][c];
                            *q++ = v;
                        }
                    }
            }
        };
        auto rows_h = [&](int r, bool inner, bool outer, const V4 &ed0, const V4 &ed2, const R *er) {
            const V4 q0 = row(3, r), q1 = row(4, r), q2 = row(5, r);
            const V4 fri = my_rad[0], frh = my_rad[1], ga = my_rad[2], gb = my_rad[3];
#pragma unroll
            for (int c = 0; c < CX; ++c) {
                // the last two rows wait for the row below (a short band's last row is its ghost)
                const bool is_inner = r + 2 < RB && c + 1 < CX;
                if (is_inner ? inner : outer) {
                    const R e0n = r + 1 < RB ? e[0][r + 1 < RB ? r + 1 : 0][c] : ed0.c[c], e2n = r + 1 < RB ? e[2][r + 1 < RB ? r + 1 : 0][c] : ed2.c[c];
                    const R e1r = c + 1 < CX ? e[1][r][c + 1 < CX ? c + 1 : 0] : er[r] * xr, e2r = c + 1 < CX ? e[2][r][c + 1 < CX ? c + 1 : 0] : er[KV * CX + r] * xr;
                    cell_h(r, c, e0n, e2n, e1r, e2r, q0, q1, q2, fri, frh, ga, gb);
                }
            }
        };
        auto read_cols = [](const V4 *from, R (&to)[2 * KV * CX]) {   // two columns, by 16-byte loads
#pragma unroll
            for (int k = 0; k < 2 * KV; ++k) {
                const V4 v = from[k];
#pragma unroll
                for (int c = 0; c < CX; ++c) to[k * CX + c] = v.c[c];
            }
        };
        auto phase_h = [&](int i) {
            if (flags & F_LATE) {   // the ragged right edge keeps the column across the wall in its first unused one
                __syncthreads();
                const R *const er = reinterpret_cast<const R *>(own + SL::ER);
                const int w = (int)((flags >> F_W) & 3u) + 1;
#pragma unroll
                for (int r = 0; r < RB; ++r)
#pragma unroll
                    for (int c = 1; c < CX; ++c)
                        if (w == c) {
                            e[1][r][c] = er[r] * bxr;
                            e[2][r][c] = er[KV * CX + r] * bxr;
                        }
            }
            V4 z{};
#pragma unroll
            for (int r = 0; r + 2 < RB; ++r) rows_h(r, true, false, z, z, nullptr);
            if (!(flags & F_LATE)) __syncthreads();
            if (EL && i > 0) consume(i - 1);
            wait_far(F_NEEDD, F_LEADD, mb_d, i);
            const V4 ed0 = own[SL::ED], ed2 = own[SL::ED + 1];
            R er[2 * KV * CX];
            read_cols(own + SL::ER, er);
            if (RB > 1) {
                const bool cut = flags & F_SHORT;
#pragma unroll
                for (int c = 0; c < CX; ++c) {
                    e[0][RB - 1][c] = cut ? ed0.c[c] : e[0][RB - 1][c];
                    e[2][RB - 1][c] = cut ? ed2.c[c] : e[2][RB - 1][c];
                }
            }
#pragma unroll
            for (int r = 0; r < RB; ++r) rows_h(r, false, true, ed0, ed2, er);
        };
        auto rows_e = [&](int r, bool inner, bool outer, const V4 &hu0, const V4 &hu2, const R *hl) {
            const V4 q0 = row(0, r), q1 = row(1, r), q2 = row(2, r);
            const V4 frh = my_rad[4], fri = my_rad[5], fa = my_rad[6], fb = my_rad[7];
#pragma unroll
            for (int c = 0; c < CX; ++c) {
                const bool is_inner = r > 0 && c > 0;
                if (is_inner ? inner : outer) {
                    const R h0p = r > 0 ? hh[0][r > 0 ? r - 1 : 0][c] : hu0.c[c], h2p = r > 0 ? hh[2][r > 0 ? r - 1 : 0][c] : hu2.c[c];
                    const R h1l = c > 0 ? hh[1][r][c > 0 ? c - 1 : 0] : hl[r] * xl, h2l = c > 0 ? hh[2][r][c > 0 ? c - 1 : 0] : hl[KV * CX + r] * xl;
                    cell_e(r, c, h0p, h2p, h1l, h2l, q0, q1, q2, frh, fri, fa, fb);
                }
            }
        };
        auto phase_e = [&](int i) {
            V4 z{};
#pragma unroll
            for (int r = 1; r < RB; ++r) rows_e(r, true, false, z, z, nullptr);
            __syncthreads();
            if (!EL && i > 0) consume(i - 1);
            wait_far(F_NEEDU, F_LEADU, mb_u, i);
            const V4 hu0 = own[SL::HU], hu2 = own[SL::HU + 1];
            R hl[2 * KV * CX];
            read_cols(own + SL::HL, hl);
#pragma unroll
            for (int r = 0; r < RB; ++r) rows_e(r, false, true, hu0, hu2, hl);
        };

        if (EL) push_e(0);
        else push_h(0);
#pragma unroll 1
        for (int i = 0; i < cnt; ++i) {
            asm volatile("" : "+r"(flags), "+r"(pk_row), "+r"(pk_col), "+r"(pk_stage));
            if (EL) {
                phase_h(i);
                push_h(i);
                phase_e(i);
                stage(i);
                if (i + 1 < cnt) push_e(i + 1);
            } else {
                phase_e(i);
                push_e(i);
                phase_h(i);
                stage(i);
                if (i + 1 < cnt) push_h(i + 1);
            }
            if (flags & F_FIRST) {   // after the half step: the first group's coefficients take their full value
                flags &= ~F_FIRST;
                if constexpr (UNI) {
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        if (EL) kH[k] *= (R)2;
                        else kE[k] *= (R)2;
                    }
                } else {
                    R *const o = reinterpret_cast<R *>(const_cast<V4 *>(ow));
#pragma unroll 1
                    for (int q = EL ? 3 * RB * CX : 0; q < (EL ? 6 : 3) * RB * CX; ++q) o[q] *= (R)2;
                }
            }
        }
        __syncthreads();
        consume(cnt - 1);
    };
    if (electric) {
        if (uni) march(ResFlag<true>{}, ResFlag<true>{});
        else march(ResFlag<false>{}, ResFlag<true>{});
    } else {
        if (uni) march(ResFlag<true>{}, ResFlag<false>{});
        else march(ResFlag<false>{}, ResFlag<false>{});
    }

    int t2 = threadIdx.x;
    asm volatile("" : "+r"(t2));
    {
        const int lb = t2 / D.tcols, tc = t2 - lb * D.tcols, b = (int)cluster_rank() * D.nb / (int)cluster_size() + lb;
        const int nx = S.n[0], ny = S.n[1];
        const int y0 = b * ny / D.nb, x0 = tc * CX, h = (flags & F_SHORT) ? RB - 1 : RB, w = (int)((flags >> F_W) & 3u) + 1;
        const unsigned N = (unsigned)nx * (unsigned)ny;
        R *const f = reinterpret_cast<R *>(S.fields);
        if (flags & F_ACTIVE) {
#pragma unroll
            for (int r = 0; r < RB; ++r)
#pragma unroll
                for (int c = 0; c < CX; ++c)
                    if (r < h && c < w) {
                        const int y = y0 + r + D.shift;
                        const unsigned g = (unsigned)((y >= ny ? y - ny : y) * nx + x0 + c);
#pragma unroll
                        for (int k = 0; k < 3; ++k) {
                            f[(unsigned)k * N + g] = e[k][r][c];
                            f[(unsigned)(3 + k) * N + g] = hh[k][r][c];
                        }
                    }
        }
    }
    if (flags & F_DEAD) *D.status = 1;
    sums.finish(D, cnt, S.acc, S.tail);
    if (flags & F_DEAD) linger();
}

}  // namespace

template <typename R, int RB>
static const void *rescyl_fn() { return (const void *)k_rescyl<R, RB, RES_MAXT>; }

const void *rescyl_kernel(int fp64, int rb)
{
    if (fp64) return rb == 1 ? rescyl_fn<double, 1>() : rb == 2 ? rescyl_fn<double, 2>() : nullptr;
    return rb == 2 ? rescyl_fn<float, 2>() : rb == 3 ? rescyl_fn<float, 3>() : nullptr;
}

int rescyl_words(int fp64, int rb, int *coef)
{
    const int cx = fp64 ? 2 : 4, kv = (rb + cx - 1) / cx;
    *coef = (6 * rb) | 1;
    return (4 + 4 * kv) | 1;
}

}  // namespace cas
