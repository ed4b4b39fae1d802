// FP64-accurate real space on the integer pipes (included by coulomb.cu, which
// defines the exact pair functions and the tile staging).
//
// Bound: the integer multiply-add pipe (a 32 x 32 + 64 bit product holds it four
// cycles: 52% busy, ALU 37%, shared-memory wavefronts 56%, 22 warps an SM), against
// 26 to 65 FP64 instructions per pair of k_real64 at 19 cycles of the SM's FP64 pipe
// each.  One block per SM takes the bricks in turn (or nchunk-ths of their rows
// where a box has few bricks); it keeps the pair table (62 KB) and, where it fits,
// the correction table (52 KB) in shared memory and stages each brick's tile there
// as fixed-point coordinates, charges and widths (40 bytes an atom).  tpr lanes
// share a row: lane l takes word l mod 4 of the row's list stripes l / 4,
// l / 4 + tpr / 4, ...
// 300,000 atoms, field: 1.49 ms (k_real64: 5.48), potential only 0.83 (3.66); the
// apply 6.31 -> 2.41 ms, 22,233 atoms at order 6 521 -> 207 us, 648 atoms 112 -> 56 us.
// Error of v, E, F against plain 64-bit sums (2-norm): 1.3e-15 at 300,000 atoms
// (k_real64: 1.2e-15), 8.8e-16 at 22,233 (8.7e-16), 8.3e-16 at 648 (9.0e-16).
// Not kept: a queue of corrections per lane instead of per row (22,233 atoms: 236
// us); corrections inline (2.07 ms at 300,000 atoms); two entries at a time without
// branches (no faster); one block per brick, staging the tables each time (1.52 ms).
#pragma once

struct FxArgs {
    int nchunk;
    int tpr_log2;               // lanes per row: 4, 8, 16 or 32
    int coord_bits, sigma_bits; // 59 - e, 56 - 2 e of the scaled lengths r' = r / 2^e
    u32 hi_cut;                 // high word of s: below it certainly inside the cutoff,
                                // above hi_cut + 2 certainly outside
    int fx_exp;                 // e
    u64 L[3];                   // box edges as coordinates
    double v_scale, e_scale;    // k_e 2^-e and k_e 2^-2e
};

// What the exact (FP64) path of one pair reads.
struct FxExact {
    RealArgs a;
    const double4_32a *xq;
    const double *sg;
    const double *erfc_tab;
    const double2 *fg_tab, *gc_tab;
};

// A pair the fixed-point path does not decide (at the cutoff to within 2^-21, or
// nearer than the pair table reaches; with corr_only, the Gaussian correction of a
// pair its table does not reach, or of a very wide charge): the arithmetic of
// k_real64, with the sorted FP64 inputs.  Adds q_j f and q_j gc d; returns f.
template <bool FIELD>
__device__ __noinline__ double fx_exact_pair(const FxExact &X, int i, int j, int code, bool corr_only,
                                           double *acc) {
    const double4_32a xi = X.xq[i];
    double4_32a xj = X.xq[j];
    xj.x += (double)(code / 25 - 2) * X.a.Lx;
    xj.y += (double)((code / 5) % 5 - 2) * X.a.Ly;
    xj.z += (double)(code % 5 - 2) * X.a.Lz;
    const double dx = xj.x - xi.x;
    const double dy = xj.y - xi.y;
    const double dz = xj.z - xi.z;
    const double r2 = dx * dx + dy * dy + dz * dz;
    if (!(r2 < X.a.rc2)) return 0.0;
    double f = 0.0, gc = 0.0;
    if (!corr_only &&
        !pw_eval<kFGShape.oct_lo, kFGShape.sub_log2, kFGShape.ncoef>(
            X.fg_tab, (unsigned)X.a.fg_pieces, r2, f, gc)) {
        const double ir = rsqrt(r2);
        double d1;
        f = erfc_pw(X.erfc_tab, X.a.alpha * (r2 * ir), d1) * ir;
        gc = (X.a.alpha * d1 - f) * ir * ir;
    }
    const double si = X.sg[i], sj = X.sg[j];
    const double si2 = si * si;
    if (r2 < kErfcXMax * kErfcXMax * (si2 + sj * sj)) {
        double fc, gcc;
        gauss_corr64(r2, si2, sj, X.erfc_tab, X.gc_tab, (unsigned)X.a.gc_pieces, fc, gcc);
        f -= fc;
        gc -= gcc;
    }
    acc[0] += xj.w * f;
    if (FIELD) {
        const double gq = xj.w * gc;
        acc[1] += gq * dx;
        acc[2] += gq * dy;
        acc[3] += gq * dz;
    }
    return f;
}

// Bytes of a tile atom: coordinates, charge (high word and fx_low), sigma^2.
constexpr size_t kFxTileBytes = 40;
constexpr int kFxThreads = 704;
constexpr int kFxQueue = 16;
constexpr size_t kFxCorrBytes = sizeof(FxRow) * kFxCorrRows;

// Charges are below 2^60, and q G keeps 5 bits below its high word (below 2^62).
constexpr int kFxQBits = 60, kFxGqUp = 5;
// Binary exponents of the high sums: F 2^-59 times q 2^(Eq - 60) times 2^64, and
// G 2^-60 q 2^(Eq - 60) 2^(64 - up) times d 2^-59 times 2^64, with Eq = e0 - 1022.
constexpr int kFxVUnit = 64 - kFxFBits - kFxQBits - 1022;
constexpr int kFxEUnit = 64 - kFxGBits - kFxQBits + 64 - kFxGqUp - kFxCoordBits - 1022;

// High sums that came near the end of their range (a crowd of atoms within half a
// scaled length) move into the row's FP64 part.
template <bool FIELD>
__device__ __noinline__ void fx_spill(FxSum &v, FxSum &ex, FxSum &ey, FxSum &ez, int e0, int fx_exp,
                                      double *acc) {
    acc[0] += scalbn((double)v.h, kFxVUnit + e0 - fx_exp);
    v.h = 0;
    if (FIELD) {
        FxSum *s[3] = {&ex, &ey, &ez};
        for (int d = 0; d < 3; ++d) {
            acc[1 + d] -= scalbn((double)s[d]->h, kFxEUnit + e0 - 2 * fx_exp);
            s[d]->h = 0;
        }
    }
}

// CORR_SMEM: the correction table is staged in shared memory too (else it is read
// through the L1 cache).
template <bool FIELD, bool CORR_SMEM>
__global__ void __launch_bounds__(kFxThreads, 1)
k_real64_fixed(const __grid_constant__ FxArgs p, const __grid_constant__ FxExact X,
               const __grid_constant__ BrickGeom g, const int4 *__restrict__ tile_tab,
               const int32_t *__restrict__ tile_tot, const uint16_t *__restrict__ nbr,
               const int32_t *__restrict__ cnt, const ulonglong4_32a *__restrict__ xfix,
               const u64 *__restrict__ sfix, const FxRow *__restrict__ pair_tab, int npair,
               const FxRow *__restrict__ corr_tab, int cap, int qcap,
               int32_t *__restrict__ flags, double *__restrict__ v_s, double *__restrict__ E_s,
               double *__restrict__ pair_f) {
    extern __shared__ __align__(32) unsigned char smem_raw[];
    __shared__ int t_start[kMaxTileBricks], t_base[kMaxTileBricks], t_code[kMaxTileBricks], t_total;
    // shared memory: pair table (npair rows), correction table, tile
    FxRow *pt = (FxRow *)smem_raw;
    FxRow *ct = pt + npair;
    ulonglong2 *tA = (ulonglong2 *)(CORR_SMEM ? ct + kFxCorrRows : ct);  // (X, Y)
    ulonglong2 *tB = tA + cap;                                                // (Z, q)
    u64 *tS = (u64 *)(tB + cap);                                              // sigma^2
    u32 *cq = (u32 *)(tS + cap);  // the rows' queues of corrections, qcap entries a lane
    {
        const uint4 *src = (const uint4 *)pair_tab;
        uint4 *dst = (uint4 *)pt;
#pragma unroll 4
        for (int t = threadIdx.x; t < npair * kFxRowWords; t += blockDim.x) dst[t] = src[t];
        if (CORR_SMEM) {
            const uint4 *sc = (const uint4 *)corr_tab;
            uint4 *dc = (uint4 *)ct;
#pragma unroll 4
            for (int t = threadIdx.x; t < kFxCorrRows * kFxRowWords; t += blockDim.x) dc[t] = sc[t];
        }
    }
    const FxRow *corr = CORR_SMEM ? ct : corr_tab;
    const int e0 = flags[kFlagChargeExp];
    const u32 smax_hi = (u32)flags[kFlagSigmaMax];
    const int lane = threadIdx.x & 31;
    const int tpr = 1 << p.tpr_log2;
    const int l = threadIdx.x & (tpr - 1);
    const int sub = l & 3, nh = tpr >> 2;
    const int rpp = blockDim.x >> p.tpr_log2;
    const size_t wstep = (size_t)kListStripe / 4 * X.a.n;  // one stripe further, in 8-byte words
    const unsigned row_mask = (tpr == 32 ? 0xffffffffu : (1u << tpr) - 1u) << (lane & ~(tpr - 1));
    const unsigned lt = (1u << lane) - 1u;
    // the row's queue: the entries that need the correction, in the order found
    u32 *rq = cq + (size_t)(threadIdx.x >> p.tpr_log2) * qcap * tpr;
    const int qfull = (qcap - 4) * tpr;  // room for one more word of every lane
    // a block keeps the tables and takes every gridDim-th unit
    for (int64_t unit = blockIdx.x; unit < g.nbricks * p.nchunk; unit += gridDim.x) {
    const int64_t b = unit / p.nchunk;
    const int chunk = (int)(unit - b * p.nchunk);
    __syncthreads();  // the previous unit's tile is no longer read
    for (int rb = threadIdx.x; rb < g.T; rb += blockDim.x) {
        const int4 e = tile_tab[b * g.T + rb];
        t_start[rb] = e.x;
        t_base[rb] = e.y;
        t_code[rb] = e.z;
    }
    if (threadIdx.x == 0) t_total = tile_tot[b];
    __syncthreads();
    const int total = t_total;
    if (total > cap) {
        if (threadIdx.x == 0) atomicExch(&flags[kFlagTileOverflow], 1);
        continue;
    }
#pragma unroll 4
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        const int rb = tile_locate(t, g.T, t_start, t_base);
        const int j = t - t_base[rb], code = t_code[rb];
        const ulonglong4_32a x = xfix[j];
        const s64 qi = fx_charge(__longlong_as_double((long long)x.w), e0, kFxQBits);
        tA[t] = make_ulonglong2(x.x + (u64)(s64)(code / 25 - 2) * p.L[0],
                                x.y + (u64)(s64)((code / 5) % 5 - 2) * p.L[1]);
        tB[t] = make_ulonglong2(x.z + (u64)(s64)(code % 5 - 2) * p.L[2],
                                ((u64)fx_hi((u64)qi) << 32) | (u32)fx_low((u64)qi));
        tS[t] = sfix[j];
    }
    __syncthreads();
    int i0, offc, nrows;
    home_rows(g, t_start, t_base, total, i0, offc, nrows);
    // this block's rows: a contiguous nchunk-th of the brick's
    const int per = (nrows + p.nchunk - 1) / p.nchunk;
    const int rbeg = chunk * per, rend = min(nrows, rbeg + per);
    for (int r0 = rbeg; r0 < rend; r0 += rpp) {
        const int r = r0 + (threadIdx.x >> p.tpr_log2);
        const bool act = r < rend;
        FxSum v, ex, ey, ez;
        double xacc[4];
        bool exact = false;
        const int rr = act ? r : rbeg, i = i0 + rr;
        const ulonglong2 ai = tA[offc + rr];
        const u64 zi = tB[offc + rr].x;
        const u64 s2i = tS[offc + rr];
        // no correction above this high word of s, whatever sigma_j is (t < 36)
        const u32 gmax = fx_hi(s2i) + smax_hi + 1;
        const u32 bound = gmax + (gmax >> 3);
        const int c = act ? cnt[i] : 0;
        // returns the pair value it added, in units of F
        auto to_exact = [&](int e, bool corr_only) {
            if (!exact) xacc[0] = xacc[1] = xacc[2] = xacc[3] = 0.0;
            exact = true;
            const int rb = tile_locate(e, g.T, t_start, t_base);
            return scalbn(fx_exact_pair<FIELD>(X, i, e - t_base[rb], t_code[rb], corr_only, xacc),
                          kFxFBits + p.fx_exp);
        };
        // kept pair values (pair_f): slot within the row's stripes as in the list
        double *row_f = pair_f ? pair_f + (size_t)i * kListStripe : nullptr;
        auto kept = [&](int pos) {
            return row_f + (size_t)(pos / kListStripe) * kListStripe * X.a.n + pos % kListStripe;
        };
        // the pair's terms from F, G 2^-b and the differences
        auto add = [&](s64 F, s64 G, u64 q, s64 dx, s64 dy, s64 dz, int lz) {
            const s32 qh = (s32)fx_hi(q), ql = (s32)fx_lo(q);
            v.add((u64)F, qh, ql);
            if (FIELD) {
                const s64 gq = fx_mul((u64)G, qh, ql, kFxGqUp);
                const s32 gh = fx_his(gq), gl = fx_low((u64)gq);
                if (lz >= 10) {  // s < 1
                    const int b = fx_bshift(lz);
                    dx <<= b;
                    dy <<= b;
                    dz <<= b;
                }
                ex.add((u64)dx, gh, gl);
                ey.add((u64)dy, gh, gl);
                ez.add((u64)dz, gh, gl);
            }
        };
        // at most four terms (each below 2^60) between folds: a high sum below 2^61
        // stays in range
        auto fold = [&]() {
            v.fold();
            u32 t = (u32)fx_his(v.h) + 0x20000000u;
            if (FIELD) {
                ex.fold();
                ey.fold();
                ez.fold();
                t |= ((u32)fx_his(ex.h) + 0x20000000u) | ((u32)fx_his(ey.h) + 0x20000000u) |
                     ((u32)fx_his(ez.h) + 0x20000000u);
            }
            if (t >= 0x40000000u) {
                if (!exact) xacc[0] = xacc[1] = xacc[2] = xacc[3] = 0.0;
                exact = true;
                FxSum tv = v, tx = ex, ty = ey, tz = ez;
                fx_spill<FIELD>(tv, tx, ty, tz, e0, p.fx_exp, xacc);
                v = tv;
                ex = tx;
                ey = ty;
                ez = tz;
            }
        };
        const uint2 *pw = (const uint2 *)(nbr + list_index(sub, i, X.a.n)) + (size_t)(l >> 2) * wstep;
        int k = (l >> 2) * kListStripe + sub;
        uint2 next = k < c ? __ldg(pw) : make_uint2(0u, 0u);
        // Pairs that need the correction (a fifth of those inside the cutoff) go to the
        // row's queue, which its lanes share out when it is full or the rows end.
        // The warp's lanes walk their words together (the ballots need them all).
        const int words = (c + nh * kListStripe - 1) / (nh * kListStripe);
        int left = __reduce_max_sync(0xffffffffu, words);
        int nq = 0;
        while (left > 0) {
            const uint2 cur = next;
            const int k0 = k;
            pw += (size_t)nh * wstep;
            k += nh * kListStripe;
            if (k < c) next = __ldg(pw);
            --left;
            u32 w0 = cur.x, w1 = cur.y;
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int e = (int)(w0 & 0xffffu);
                w0 = __funnelshift_r(w0, w1, 16);
                w1 >>= 16;
                bool queue = false;
                // the entry's place in the row (stripe, lane's word, entry)
                const int pos = (k0 & ~(kListStripe - 1)) + sub * 4 + u;
                double kf = 0.0;
                // past the row's end (padding entries are e = total)
                if (k0 + kListLanes * u < c && e < total) {
                    const ulonglong2 aj = tA[e];
                    const ulonglong2 bj = tB[e];
                    const s64 dx = (s64)(aj.x - ai.x), dy = (s64)(aj.y - ai.y), dz = (s64)(bj.x - zi);
                    const u64 s = fx_dist2(dx, dy, dz);
                    const u32 sh = fx_hi(s);
                    if (sh <= p.hi_cut + 2) {
                        const int lz = fx_clz(sh);
                        if (sh < p.hi_cut && lz <= kFxLzMin) {
                            const u64 y = fx_pos(s, lz);
                            u64 F, G = 0;
                            fx_eval<FIELD, kFxGShift>(pt[fx_piece(sh, lz)], fx_hi(y), fx_lo(y), F, G);
                            add((s64)F, (s64)G, bj.y, dx, dy, dz, lz);
                            if (row_f) kf = (double)F;
                            if ((sh >> 3) < bound) {
                                const u32 gh = fx_hi(s2i + tS[e]);
                                queue = (sh >> 3) < gh + (gh >> 3);
                            }
                        } else {
                            kf = to_exact(e, false);
                        }
                    }
                }
                if (row_f && k0 < c) *kept(pos) = kf;
                const unsigned m = __ballot_sync(0xffffffffu, queue) & row_mask;
                if (queue) rq[nq + __popc(m & lt)] = (u32)e | (u32)pos << 16;
                nq += __popc(m);
            }
            fold();
            if (left > 0 && !__any_sync(0xffffffffu, nq > qfull)) continue;
            __syncwarp();
            for (int m = l; m < nq; m += tpr) {
                const u32 qe = rq[m];
                const int e = (int)(qe & 0xffffu);
                const ulonglong2 aj = tA[e];
                const ulonglong2 bj = tB[e];
                const s64 dx = (s64)(aj.x - ai.x), dy = (s64)(aj.y - ai.y), dz = (s64)(bj.x - zi);
                const u64 s = fx_dist2(dx, dy, dz);
                const int lz = fx_clz(fx_hi(s));
                const u64 g2 = s2i + tS[e];
                s64 F = 0, G = 0;
                if (g2 < kFxSigmaSat && fx_correct<FIELD>(corr, s, fx_bshift(lz), g2, F, G)) {
                    add(F, G, bj.y, dx, dy, dz, lz);
                    fold();
                    if (row_f) *kept((int)(qe >> 16)) += (double)F;
                } else {
                    const double kf = to_exact(e, true);
                    if (row_f) *kept((int)(qe >> 16)) += kf;
                }
            }
            nq = 0;
            __syncwarp();
        }
        // lanes of the row: integer sums (32 of them must fit: five bits of the high
        // sum move to the cross sum first), then one lane per component converts
        auto lanes = [&](FxSum &q) {
            q.m += (q.h & 31) << kFxCross;
            q.h >>= 5;
            for (int o = 1; o < tpr; o <<= 1) {
                q.h += __shfl_xor_sync(0xffffffffu, q.h, o);
                q.m += __shfl_xor_sync(0xffffffffu, q.m, o);
            }
        };
        lanes(v);
        if (FIELD) {
            lanes(ex);
            lanes(ey);
            lanes(ez);
        }
        double extra = 0.0;  // exact pairs' part of this lane's component
        if (__any_sync(0xffffffffu, exact)) {
#pragma unroll
            for (int d = 0; d < (FIELD ? 4 : 1); ++d) {
                double t = exact ? xacc[d] : 0.0;
                for (int o = 1; o < tpr; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                if (l == d) extra = t;
            }
        }
        if (act && l < (FIELD ? 4 : 1)) {
            const s64 h = l == 0 ? v.h : l == 1 ? ex.h : l == 2 ? ey.h : ez.h;
            const s64 m = l == 0 ? v.m : l == 1 ? ex.m : l == 2 ? ey.m : ez.m;
            const double sum = scalbn(fma((double)h, (double)(1ll << (kFxCross + 5)), (double)m),
                                      (l == 0 ? kFxVUnit : kFxEUnit) + e0 - kFxCross);
            if (l == 0)
                v_s[i] = fma(X.a.ke, extra, p.v_scale * sum);
            else
                E_s[3 * (size_t)i + (l - 1)] = fma(X.a.ke, extra, -(p.e_scale * sum));
        }
    }
    }
}

// Launch of the fixed-point kernel for the current list: on = false where its tile
// and pair table exceed a block's shared memory (then k_real64 runs).
struct FxLaunch {
    bool on;
    bool corr_smem;
    int threads, nchunk, tpr_log2, npair;
    int qcap;  // entries of a lane's correction queue
    u32 hi_cut;
    size_t smem;
};

inline FxLaunch fx_launch(const qeq_ctx *ctx) {
    FxLaunch L{};
    if (!ctx->fx_on) return L;
    const double rc = std::ldexp(ctx->p.r_cut, -ctx->fx_exp);
    L.hi_cut = (u32)std::floor(std::ldexp(rc * rc, 22)) - 1u;
    L.npair = fx_piece(L.hi_cut, fx_clz(L.hi_cut)) + 1;
    // blocks per brick: the fewest waves of one block per SM, a block's time being
    // its rows plus about 0.15 of a brick for staging its tile
    const int64_t nb = ctx->geom.nbricks;
    const int rows = std::max(1, ctx->rows_cap);
    double best = 0.0;
    for (int c = 1; c <= 8 && (c == 1 || c * 4 <= rows); ++c) {
        const double cost = (double)((nb * c + ctx->sm_count - 1) / ctx->sm_count) * (1.0 / c + 0.15);
        if (c == 1 || cost < best) {
            best = cost;
            L.nchunk = c;
        }
    }
    // lanes per row: as many as the block holds for its rows
    const int per = (rows + L.nchunk - 1) / L.nchunk;
    L.tpr_log2 = 2;
    while (L.tpr_log2 < 5 && (per << (L.tpr_log2 + 1)) <= kFxThreads) ++L.tpr_log2;
    const int want = ((per << L.tpr_log2) + 31) / 32 * 32;
    L.threads = std::min(kFxThreads, std::max(512, want));  // idle warps still stage the tile
    // shared memory: the pair table, the tile and the shortest queues must fit; the
    // correction table comes in where it leaves room for them, the queues take up
    // to kFxQueue entries of the rest
    const size_t slot = sizeof(u32) * L.threads;
    const size_t base = sizeof(FxRow) * L.npair + (size_t)ctx->tile_cap * kFxTileBytes;
    if (base + 4 * slot > kReal64SmemMax) return L;
    L.corr_smem = base + kFxCorrBytes + 4 * slot <= kReal64SmemMax;
    L.smem = base + (L.corr_smem ? kFxCorrBytes : 0);
    L.qcap = (int)std::min<size_t>(kFxQueue, (kReal64SmemMax - L.smem) / slot);
    L.smem += L.qcap * slot;
    L.on = true;
    return L;
}
