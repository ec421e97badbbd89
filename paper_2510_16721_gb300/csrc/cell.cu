// Cell filter inverse map and cell-list build.
//
// Map-back (Sec. II.C): the lattice rows of X hold c B; B = X_lat / c is
// symmetrised and D = B^(1/2) taken with a coupled Newton-Schulz iteration in FP64
// (rotation-free variant), or D = X_lat / c (deformation-gradient variant).
// Then h = h0 D, and the bin geometry of the image is derived from the
// perpendicular widths of h.
//
// Cell list: atoms are binned in fractional space (s = R~ h0^-1, which is
// also R h^-1 since R = R~ D and h = h0 D), wrapped into [0, 1).  The bin
// edge vectors bv_a = h_a / nb_a are rounded to T, and each atom stores its
// Cartesian offset from the centre of its bin, sum_a (b_a + 1/2) bv_a, in T.
// A pair vector is then (off_j - off_i) + sum_a (delta_a bv_a + t_a dh_a),
// where delta is the unwrapped bin offset of the neighbour bin, t its
// periodic shift and dh_a = h_a - nb_a bv_a the (tiny) difference between a
// lattice vector and nb_a rounded bin vectors.  For |delta| <= 1 in an
// orthorhombic cell every term is exact in FP32, so the only roundings are
// those of the two small offsets and of the final sums: pair vectors keep
// ~6e-8 A absolute accuracy whatever the cell size.  (FP32 many-body bands store
// integer grid positions instead, see refresh_offset.)  Enumerating delta over
// [-m_a, m_a] with m_a = ceil(rc / bin width) visits every periodic image
// of every atom within rc exactly once, also when rc exceeds half the cell
// width (no minimum-image assumption; the neighbourhoods of Sec. II.B are
// periodic).
//
// Determinism: atoms are counted into bins with integer atomics, then each
// bin's atoms are ordered by atom index, so the slot order (and every
// summation order downstream) is the same on every run.
//
// Reuse with a skin: with skin > 0 the stencil and any neighbour list cover
// rl = rc + skin, and an image keeps its bins (and lists) while they still
// hold every pair inside rc.  With R = R~ D, a pair vector is rho D where
// rho is its R~-frame vector; from the build (D_b) to now (D), a pair that
// was at |r_b| >= rl is now at least rl (1 - |D_b^-1 D - I|) - 2 d |D| away,
// d being the largest displacement |R~ - R~_b| of any atom.  While that
// bound stays above rc the bins of the build are kept: each atom's offset is
// recomputed from its current position against the centre of its old bin
// (the pair-vector identity above holds for any position, inside the bin or
// not), which costs one pass over the atoms instead of a rebuild.
#include <algorithm>

#include "common.cuh"

namespace cfneb {

// ---- 3x3 symmetric square root -----------------------------------------
//
// On this GPU a dependent FP64 operation costs ~64 cycles and an FP64
// divide or square root several hundred, and the map-back of every image is
// on the critical path of each step.  The symmetric root is therefore taken
// with the coupled Newton-Schulz iteration (Higham, Functions of Matrices,
// 2008, Sec. 6.7), which needs matrix products only: with Y0 = B/mu, Z0 = I
// and T = (3I - Z Y)/2, Y <- Y T and Z <- T Z converge quadratically to
// (B/mu)^(1/2) and (B/mu)^(-1/2) when the eigenvalues of B/mu lie in (0, 2).
// Every iterate is a polynomial in B, so Y and Z stay symmetric and commute
// with B.  mu is the midpoint of a bracket of the spectrum: g, the largest
// Gershgorin row bound (>= lambda_max), and det B / g^2 (<= lambda_min).
// The products run lane-parallel (k_mapback).

// Bin grid of an image with cell h (one thread): the bin counts nb and
// stencil half widths m from the perpendicular widths and the list cutoff.
// Between rebuilds the grid stays as built and only the bin vectors follow
// the cell (bin_vectors_warp).
// status: the band's word in memory (bp may be a staged copy).
__device__ void bin_grid(const BandParams *bp, int nbins_cap, const double *h, double omega,
                         ImgScalars &sc, int *status) {
    const double rl = bp->rl > 0.0 ? bp->rl : bp->rc;
    int nb[3];
    float w[3];
    // perpendicular widths w_a = Omega / |h_b x h_c| (only choose the bin
    // grid: FP32, shaded down by 1e-4 so the stencil is never too narrow,
    // also for atoms binned in FP32)
    for (int a = 0; a < 3; ++a) {
        const double *u = h + 3 * ((a + 1) % 3), *v = h + 3 * ((a + 2) % 3);
        const double cx = u[1] * v[2] - u[2] * v[1], cy = u[2] * v[0] - u[0] * v[2],
                     cz = u[0] * v[1] - u[1] * v[0];
        w[a] = (float)omega / sqrtf((float)(cx * cx + cy * cy + cz * cz)) * 0.9999f;
        // a cell whose volume or areas leave FP32's range: refused, and on with a
        // grid that is safe (a NaN here would give no bin at all, and the walks
        // that wrap by the bin count would not end)
        if (!(w[a] > 0.0f && w[a] <= 3e38f)) {
            atomicOr(status, ST_NBR_OVERFLOW);
            w[a] = (float)rl;
        }
    }
    for (int a = 0; a < 3; ++a) {
        // the innermost axis may be binned finer: the LJ kernel walks it
        // as contiguous rows, so finer bins there trim the candidate
        // range without adding rows
        const float bw = (float)bp->bin_w / (a == 2 ? (float)bp->row_refine : 1.0f);
        // never so fine that the stencil would need more than
        // MAX_STENCIL bins per side (coarser bins are always correct)
        const float q = fminf(floorf(w[a] / bw),
                              floorf(w[a] * (float)MAX_STENCIL / (float)rl * 0.9999f));
        nb[a] = q >= 1.0f ? (q > 1024.0f ? 1024 : (int)q) : 1;
    }
    // keep within the bin capacity: coarser bins are always correct
    while ((long long)nb[0] * nb[1] * nb[2] > nbins_cap) {
        int a = (nb[0] >= nb[1] && nb[0] >= nb[2]) ? 0 : (nb[1] >= nb[2] ? 1 : 2);
        nb[a] -= 1;
    }
    for (int a = 0; a < 3; ++a) {
        const float bw = w[a] / nb[a];
        const int m = (int)ceilf((float)rl / bw);
        // a cell narrower than rl / MAX_STENCIL: periodic images beyond the
        // stencil would be missed
        if (m > MAX_STENCIL) atomicOr(status, ST_NBR_OVERFLOW);
        sc.m[a] = m < 1 ? 1 : (m > MAX_STENCIL ? MAX_STENCIL : m);
        sc.nb[a] = nb[a];
    }
    sc.nbins = nb[0] * nb[1] * nb[2];
}

// The rebuild decision of one image on its staged record sc (one thread):
// keep the bins of the build while the bound in the header comment holds,
// else rebuild (always when forced, when the band's images were rearranged,
// or while autotuning).  d = the largest displacement since the build; the
// cell's part of the bound (skin_terms) is current in sc.
__device__ void skin_decide_one(const BandParams *bp, int nbins_cap, ImgScalars &sc, double d,
                                int force, int *status) {
    bool rebuild = force || bp->stale || bp->tune_rebuild || sc.builds == 0;
    if (!rebuild) {
        const double bound = bp->rl * (1.0 - 1e-5) * (1.0 - (double)sc.skin_e) -
                             2.0 * d * (double)sc.skin_nD * (1.0 + 1e-5);
        rebuild = !(bound > bp->rc);
    }
    if (rebuild) {
        bin_grid(bp, nbins_cap, sc.h, sc.omega, sc, status);
        float Db[9];
        for (int k = 0; k < 9; ++k) {
            sc.Db[k] = sc.D[k];
            Db[k] = (float)sc.D[k];
        }
        inv3f(Db, sc.Dbif);
        skin_terms(sc, sc.Dbif);
        sc.builds += 1;
    }
    sc.rebuild = rebuild ? 1 : 0;
    sc.dmax = d;
    sc.evals += 1;
}

// Map-back of one image per warp and its cell-list decision.  The cell
// (image_cell_warp: D, h, Omega and the bin vectors) is taken over from the
// last move when k_fire_update already computed it for the current lattice
// rows; it is computed here for forced evaluations, after the band's images
// were rearranged or reloaded (stale) and whenever the move did not leave
// it.  Then with no skin a rebuild on the new cell, with a skin the reuse
// test on the displacements the last move left per row tile.  The image
// record is staged in shared memory, updated and written back whole.
template <typename T>
__global__ void __launch_bounds__(32) k_mapback(const ImgRef *imgs, int count, BandDev *bands,
                                                int force_) {
    const ImgRef r = imgs[blockIdx.x];
    const BandDev b = bands[r.band];
    dep_sync();
    const bool force =
        force_ == REBUILD_ALL || (force_ == REBUILD_ENDS && (r.img == 0 || r.img == b.bp->N - 1));
    __shared__ BandParams s_bp;
    __shared__ ImgScalars s_sc;
    stage_copy(&s_bp, b.bp);
    stage_copy(&s_sc, &b.sc[r.img]);
    __syncwarp();
    const BandParams *bp = &s_bp;
    ImgScalars &sc = s_sc;
    const int lane = threadIdx.x & 31;
    const bool fresh = !force && !bp->stale && sc.cell_fresh;
    double h = 0.0;
    if (!fresh) {
        const T *Xl = (const T *)b.X + ((size_t)r.img * b.rows + b.n) * 3;
        const bool ok = image_cell_warp(cell_in(bp), (double)Xl[lane % 9], sc, h);
        if (!ok && lane == 0) atomicOr(&b.bp->status, ST_NOT_SPD);
    }
    // largest displacement since the last build (skin > 0), in FP32 (a max
    // is exact in any precision)
    double dmax = 0.0;
    if (b.skin_part) {
        // per row tile, left by the last move (k_fire_update)
        const float *part = b.skin_part + (size_t)r.img * b.rtpi;
        float m = 0.0f;
#pragma unroll 8
        for (int t = lane; t < b.rtpi; t += 32) m = fmaxf(m, part[t]);
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        dmax = (double)m;
    }
    __syncwarp();
    if (lane == 0) {
        sc.cell_fresh = 1;
        if (!fresh && bp->skin > 0.0) skin_terms(sc, sc.Dbif);
        if (bp->skin <= 0.0) {
            // no skin: the cell list is rebuilt at every evaluation
            bin_grid(bp, b.nbins_cap, sc.h, sc.omega, sc, &b.bp->status);
            sc.rebuild = 1;
            sc.builds += 1;
            sc.evals += 1;
        } else {
            skin_decide_one(bp, b.nbins_cap, sc, dmax, force, &b.bp->status);
        }
    }
    __syncwarp();
    // the grid (new or kept) follows the cell; a move that left the cell
    // also left the bin vectors of the kept grid
    if (!fresh || sc.rebuild) bin_vectors_warp(sc, sc.nb[(lane % 9) / 3], sc.h[lane % 9]);
    if (sizeof(T) == 4 && !fresh && b.shift)
        grid_warp(sc, b.shift + (size_t)r.img * SHIFTS * 6, sc.h[lane % 9], (float)bp->rl);
    __syncwarp();
    stage_copy(&b.sc[r.img], &s_sc);
}

// Offset of an atom from the centre of its (kept) bin, R - K with R = R~ D
// and K = sum_a (wrap_a h_a + (b_a + 1/2) bv_a), as a leading part and a
// remainder.  FP64 path: in FP64.  FP32 path: in pairs of FP32 (products
// split exactly with FMA, sums with Knuth's two-sum), from the FP32 pairs
// of D and h that k_mapback stores; bv is exact in FP32 by construction.
// Both keep the offset to ~1e-14 relative of the cell size, far below the
// FP32 leading part's rounding.  FP64 bands get the FP32 copy in lo.
__device__ inline void refresh_offset(const ImgScalars &sc, const BandParams *bp, const double *X,
                                      const int *wr, const int *bi, int, const int *,
                                      double4_32a &o, float4 &lo) {
    double off[3];
    double s[3];
    for (int a = 0; a < 3; ++a)
        s[a] = (X[0] * bp->h0inv[a] + X[1] * bp->h0inv[3 + a] + X[2] * bp->h0inv[6 + a]) -
               (double)wr[a];
    for (int c = 0; c < 3; ++c) {
        const double R = s[0] * sc.h[c] + s[1] * sc.h[3 + c] + s[2] * sc.h[6 + c];
        const double ctr = (bi[0] + 0.5) * sc.bv[c] + (bi[1] + 0.5) * sc.bv[3 + c] +
                           (bi[2] + 0.5) * sc.bv[6 + c];
        off[c] = R - ctr;
    }
    o.x = off[0];
    o.y = off[1];
    o.z = off[2];
    o.w = (double)bi[2];
    lo = make_float4((float)off[0], (float)off[1], (float)off[2], (float)bi[2]);
}

__device__ inline F2 f2_prod(float a, float b) {  // a b exactly
    const float p = __fmul_rn(a, b);
    return {p, fmaf(a, b, -p)};
}

// K = sum_a (wrap_a h_a + (b_a + 1/2) bv_a) is formed as
// sum_a m_a bv_a + sum_a wrap_a dh_a with m_a = wrap_a nb_a + b_a + 1/2
// (h_a = nb_a bv_a + dh_a): each m_a bv_a is exact as a pair (bv exact in
// FP32, m_a a half-integer far below 2^23), the dh terms are tiny and join
// the low part.
//
// Many-body (Tersoff, NEP-style) bands hold the position in the cell, R -
// sum_a wrap_a h_a, on the image's integer grid instead (see
// common.cuh; o carries the integers' bits; wk: the wrap's place in the table
// of lattice shifts, SHIFTS / 2 for none, SHIFTS for one beyond the table).
__device__ inline int wrap_place(const int *wr) {
    if ((unsigned)(wr[0] + 1) > 2u || (unsigned)(wr[1] + 1) > 2u || (unsigned)(wr[2] + 1) > 2u)
        return SHIFTS;
    return (wr[0] + 1) + 3 * (wr[1] + 1) + 9 * (wr[2] + 1);
}
__device__ inline void refresh_offset(const ImgScalars &sc, const BandParams *bp, const float *X,
                                      const int *wr, const int *bi, int wk, const int *shift,
                                      float4 &o, float4 &lo) {
    if (bp->kind != KIND_LJ) {
        const float *Dh = sc.dfl, *Dl = sc.dfl + 9, *hh = sc.dfl + 18, *hl = sc.dfl + 27;
        const float g = sc.grid, ig = sc.igrid;
        int i[3];
        float l[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            F2 R = f2_mul(X[0], Dh[c], Dl[c]);
            R = f2_add(R, f2_mul(X[1], Dh[3 + c], Dl[3 + c]));
            R = f2_add(R, f2_mul(X[2], Dh[6 + c], Dl[6 + c]));
            if (wk == SHIFTS) {  // wrapped by more than a cell
#pragma unroll
                for (int a = 0; a < 3; ++a)
                    R = f2_add(R, f2_mul(-(float)wr[a], hh[3 * a + c], hl[3 * a + c]));
            }
            grid_split(R, g, ig, i[c], l[c]);
            if (wk < SHIFTS && wk != SHIFTS / 2) {  // by at most one: the table's shift
                i[c] -= shift[6 * wk + c];
                l[c] -= __int_as_float(shift[6 * wk + 3 + c]);
            }
        }
        o = make_float4(__int_as_float(i[0]), __int_as_float(i[1]), __int_as_float(i[2]), 0.0f);
        lo = make_float4(l[0], l[1], l[2], 0.0f);
        return;
    }
    const float *Dh = sc.dfl, *Dl = sc.dfl + 9;
    float m[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) m[a] = (float)(wr[a] * sc.nb[a] + bi[a]) + 0.5f;
    float off[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        // R_c = sum_k X_k D_kc (X exact in FP32)
        F2 R = f2_mul(X[0], Dh[c], Dl[c]);
        R = f2_add(R, f2_mul(X[1], Dh[3 + c], Dl[3 + c]));
        R = f2_add(R, f2_mul(X[2], Dh[6 + c], Dl[6 + c]));
        F2 K = f2_prod(m[0], sc.bvf[c]);
        K = f2_add(K, f2_prod(m[1], sc.bvf[3 + c]));
        K = f2_add(K, f2_prod(m[2], sc.bvf[6 + c]));
        K.lo = fmaf((float)wr[0], sc.dhf[c],
                    fmaf((float)wr[1], sc.dhf[3 + c], fmaf((float)wr[2], sc.dhf[6 + c], K.lo)));
        const F2 d = f2_add(R, {-K.hi, -K.lo});
        off[0][c] = d.hi;
        off[1][c] = d.lo;
    }
    o = make_float4(off[0][0], off[0][1], off[0][2], (float)bi[2]);
    lo = make_float4(off[1][0], off[1][1], off[1][2], 0.0f);
}

// A slot's position: in FP32 many-body bands one record of both parts, stored and
// loaded whole (98,303 atoms x 9 images, site terms: 59.2 us with two arrays, 55.2
// with records).
__device__ inline void store_pos(const BandDev &b, size_t st, const float4 &o, const float4 &lo) {
    if (b.shift) {
        asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                         (float4 *)b.slot_off + 2 * st),
                     "f"(o.x), "f"(o.y), "f"(o.z), "f"(o.w), "f"(lo.x), "f"(lo.y), "f"(lo.z),
                     "f"(lo.w)
                     : "memory");
    } else {
        ((float4 *)b.slot_off)[st] = o;
        b.slot_off_lo[st] = lo;
    }
}
__device__ inline void store_pos(const BandDev &b, size_t st, const double4_32a &o,
                                 const float4 &lo) {
    ((double4_32a *)b.slot_off)[st] = o;
    b.slot_off_lo[st] = lo;
}

// Bin and periodic wrap of an atom: s = R~ h0^-1 wrapped into [0, 1).  FP64
// path in FP64; FP32 path in FP32 (a bin choice off by FP32 rounding near a
// bin face puts the atom ~1e-7 of the cell outside its bin, inside the
// 1e-4 margin the stencil widths are shaded by; the offset itself is exact).
__device__ inline void bin_of(const ImgScalars &sc, const BandParams *bp, const double *X, int *bi,
                              int *wrap) {
    for (int a = 0; a < 3; ++a) {
        double s = X[0] * bp->h0inv[a] + X[1] * bp->h0inv[3 + a] + X[2] * bp->h0inv[6 + a];
        const double fl = floor(s);
        s -= fl;
        wrap[a] = (int)fl;
        if (s >= 1.0) {
            s = 0.0;
            wrap[a] += 1;
        }
        // any bin index outside [0, nb) (a non-finite coordinate) goes to an
        // edge bin: the index stays in range whatever the input
        const int q = (int)(s * sc.nb[a]);
        bi[a] = q >= sc.nb[a] ? sc.nb[a] - 1 : (q < 0 ? 0 : q);
    }
}
__device__ inline void bin_of(const ImgScalars &sc, const BandParams *, const float *X, int *bi,
                              int *wrap) {
    const float *hi = sc.dfl + 36;  // h0^-1 in FP32
    for (int a = 0; a < 3; ++a) {
        float s = X[0] * hi[a] + X[1] * hi[3 + a] + X[2] * hi[6 + a];
        const float fl = floorf(s);
        s -= fl;
        wrap[a] = (int)fl;
        if (s >= 1.0f) {
            s = 0.0f;
            wrap[a] += 1;
        }
        const int q = (int)(s * (float)sc.nb[a]);
        bi[a] = q >= sc.nb[a] ? sc.nb[a] - 1 : (q < 0 ? 0 : q);
    }
}

// In a graph (has_cond), the first tile of every image that rebuilds also
// switches on the conditional node that holds the rebuild kernels (its
// value is reset to 0 at every launch of the graph).
// FP32: 12 blocks per SM (40 registers, 18.4 us at 98,303 atoms x 9 images; 18.9
// with the 48 that the tables read ahead take).  Where the force kernel's tiles hold
// few atoms, large sets put an atom on every thread (500 FP64 bands of 31 atoms x 5
// images, tiles of 4: 62 us with a tile's atoms per block, 29 so), small ones a tile's
// atoms on a block (2,915 FP64 atoms x 5 images, tiles of 32: 10.2 us, 12.8 packed).
template <typename T>
__global__ void __launch_bounds__(TILE, sizeof(T) == 4 ? 12 : 8)
    k_bin_assign(const Tile *tiles, BandDev *bands, cudaGraphConditionalHandle cond,
                 int has_cond) {
    using T4 = typename Vec4<T>::type;
    const Tile tl = tiles[blockIdx.x];
    const BandDev b = bands[tl.band];
    dep_sync();
    const ImgScalars &sc = b.sc[tl.img];
    const BandParams *bp = b.bp;
    if (has_cond && sc.rebuild && tl.t == 0 && threadIdx.x == 0) cudaGraphSetConditional(cond, 1u);
    if (!sc.rebuild) {
        // keep the bins of the build: thread = slot, offset from the centre
        // of the slot's bin at the current position (unwrapped as at the build)
        const int t = block_atom(b, tl);
        if (t >= b.n) return;
        const size_t st = (size_t)tl.img * b.n + t;
        const int i = b.slot_atom[st];
        int bi[3] = {0, 0, 0};
        const int *wr = b.atom_wrap + ((size_t)tl.img * b.n + i) * 3;
        int wk = 0;
        if (b.shift) wk = b.slot_wrap[st];  // grid positions need no bin, and the wrap's place
        else unpack_bin(b.slot_bin[st], bi[0], bi[1], bi[2]);
        const T *Xi = (const T *)b.X + ((size_t)tl.img * b.rows + i) * 3;
        T4 o;
        float4 lo;
        refresh_offset(sc, bp, Xi, wr, bi, wk, b.shift + (size_t)tl.img * SHIFTS * 6, o, lo);
        store_pos(b, st, o, lo);
        return;
    }
    // (through the table: what only a rebuild needs holds no registers above)
    const BandDev &br = bands[tl.band];
    const int i = block_atom(br, tl);
    if (i >= br.n) return;
    const T *Xi = (const T *)br.X + ((size_t)tl.img * br.rows + i) * 3;
    int bi[3], wrap[3];
    bin_of(sc, bp, Xi, bi, wrap);
    int lin = (bi[0] * sc.nb[1] + bi[1]) * sc.nb[2] + bi[2];
    size_t ai = (size_t)tl.img * br.n + i;
    int rank = atomicAdd(&br.bin_count[(size_t)tl.img * br.nbins_cap + lin], 1);
    br.atom_bin[ai] = lin;
    br.atom_rank[ai] = rank;
    // offset from the bin centre (the w lane holds the innermost bin index,
    // for the row traversal of the LJ kernel)
    T4 o;
    float4 lo;
    refresh_offset(sc, bp, Xi, wrap, bi, wrap_place(wrap), br.shift + (size_t)tl.img * SHIFTS * 6, o,
                   lo);
    ((T4 *)br.atom_off)[ai] = o;
    br.atom_off_lo[ai] = lo;
    if (br.ref_X) {  // a skin: reference state of the build (row layout of X)
        T *ref = (T *)br.ref_X + ((size_t)tl.img * br.rows + i) * 3;
        ref[0] = Xi[0];
        ref[1] = Xi[1];
        ref[2] = Xi[2];
        for (int a = 0; a < 3; ++a) br.atom_wrap[ai * 3 + a] = wrap[a];
    }
}

// Exclusive scan of the bin counts, in three passes over SCAN_TILE-bin
// tiles: tile sums, a scan of the tile sums per image, and a block-wide scan
// of each tile offset by its tile prefix.  Integer arithmetic: exact and
// deterministic.  Counts are reset to zero for the next build.
constexpr int SCAN_TILE = 1024;

__device__ inline int block_excl_scan_1024(int v, int *total) {
    __shared__ int wsum[32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    int x = v;
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = wsum[lane];
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        wsum[lane] = s;  // inclusive scan of the warp sums
    }
    __syncthreads();
    const int before = (w > 0) ? wsum[w - 1] : 0;
    *total = wsum[31];
    __syncthreads();
    return before + x - v;
}

__global__ void __launch_bounds__(256) k_bin_tilesum(const ImgRef *imgs, BandDev *bands) {
    dep_sync();
    ImgRef r = imgs[blockIdx.x];
    BandDev &b = bands[r.band];
    if (!b.sc[r.img].rebuild) return;
    const int nb = b.sc[r.img].nbins;
    const int *cnt = b.bin_count + (size_t)r.img * b.nbins_cap;
    __shared__ int ws[8];
    // a fixed grid strides over the tiles: images that keep their cell list
    // cost one read per block
    for (int c = blockIdx.y; c * SCAN_TILE < nb; c += gridDim.y) {
        const int t0 = c * SCAN_TILE;
        int s = 0;
        for (int k = threadIdx.x; k < SCAN_TILE && t0 + k < nb; k += blockDim.x) s += cnt[t0 + k];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = s;
        __syncthreads();
        if (threadIdx.x == 0) {
            int tot = 0;
            for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tot += ws[q];
            b.bin_tsum[(size_t)r.img * b.tsum_cap + c] = tot;
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(1024) k_bin_tilescan(const ImgRef *imgs, BandDev *bands) {
    dep_sync();
    ImgRef r = imgs[blockIdx.x];
    BandDev &b = bands[r.band];
    if (!b.sc[r.img].rebuild) return;
    const int nt = (b.sc[r.img].nbins + SCAN_TILE - 1) / SCAN_TILE;
    int *ts = b.bin_tsum + (size_t)r.img * b.tsum_cap;
    int carry = 0;
    for (int base = 0; base < nt; base += 1024) {
        const int k = base + threadIdx.x;
        const int v = k < nt ? ts[k] : 0;
        int tot;
        const int ex = block_excl_scan_1024(v, &tot);
        if (k < nt) ts[k] = carry + ex;
        carry += tot;
    }
}

__global__ void __launch_bounds__(1024) k_bin_scanfill(const ImgRef *imgs, BandDev *bands) {
    dep_sync();
    ImgRef r = imgs[blockIdx.x];
    BandDev &b = bands[r.band];
    if (!b.sc[r.img].rebuild) return;
    const int nb = b.sc[r.img].nbins;
    int *cnt = b.bin_count + (size_t)r.img * b.nbins_cap;
    int *start = b.bin_start + (size_t)r.img * (b.nbins_cap + 1);
    for (int c = blockIdx.y; c * SCAN_TILE < nb; c += gridDim.y) {
        const int bin = c * SCAN_TILE + threadIdx.x;
        const int v = bin < nb ? cnt[bin] : 0;
        int tot;
        const int ex = block_excl_scan_1024(v, &tot);
        const int off = b.bin_tsum[(size_t)r.img * b.tsum_cap + c];
        if (bin < nb) {
            start[bin] = off + ex;
            cnt[bin] = 0;
            if (bin == nb - 1) start[nb] = off + ex + v;
        }
    }
}

__global__ void __launch_bounds__(TILE) k_bin_scatter(const Tile *tiles, int ntiles, BandDev *bands) {
    dep_sync();
    for (int k = blockIdx.x; k < ntiles; k += gridDim.x) {
        const Tile tl = tiles[k];
        BandDev &b = bands[tl.band];
        if (!b.sc[tl.img].rebuild) continue;
        const int i = tile_atom(b, tl);
        if (i >= b.n) continue;
        const size_t ai = (size_t)tl.img * b.n + i;
        const int *start = b.bin_start + (size_t)tl.img * (b.nbins_cap + 1);
        b.slot_unsorted[(size_t)tl.img * b.n + start[b.atom_bin[ai]] + b.atom_rank[ai]] = i;
    }
}

// Atom i of an image (whose arrays begin at base) takes slot dst of bin pb.
template <typename T>
__device__ inline void order_atom(const BandDev &b, size_t base, int i, int dst, int pb,
                                  const typename Vec4<T>::type &o, const float4 &ol) {
    b.slot_atom[base + dst] = i;
    b.slot_bin[base + dst] = pb;
    b.atom_slot[base + i] = dst;
    store_pos(b, base + dst, o, ol);
    if (b.slot_wrap) b.slot_wrap[base + dst] = wrap_place(b.atom_wrap + (base + i) * 3);
}

// Order each bin's atoms by atom index and write the sorted slot arrays: one
// thread per atom, its rank among its bin's atoms counted from the unordered
// slots.  (One thread per bin left the chip to a few threads with quadratic
// loops: 19,380 atoms in 972 bins, 54 us.)
template <typename T>
__global__ void __launch_bounds__(TILE) k_bin_order(const Tile *tiles, int ntiles, BandDev *bands) {
    dep_sync();
    using T4 = typename Vec4<T>::type;
    for (int k = blockIdx.x; k < ntiles; k += gridDim.x) {
        const Tile tl = tiles[k];
        BandDev &b = bands[tl.band];
        const ImgScalars &sc = b.sc[tl.img];
        if (!sc.rebuild) continue;
        const int i = tile_atom(b, tl);
        if (i >= b.n) continue;
        const size_t base = (size_t)tl.img * b.n;
        const int *start = b.bin_start + (size_t)tl.img * (b.nbins_cap + 1);
        const int *un = b.slot_unsorted + base;
        const int nb1 = sc.nb[1], nb2 = sc.nb[2];
        const int bin = b.atom_bin[base + i];
        const T4 o = ((const T4 *)b.atom_off)[base + i];
        const float4 ol = b.atom_off_lo[base + i];
        const int s0 = start[bin], s1 = start[bin + 1];
        int dst = s0;
        for (int q = s0; q < s1; ++q) dst += un[q] < i;
        order_atom<T>(b, base, i, dst, pack_bin(bin / (nb1 * nb2), (bin / nb2) % nb1, bin % nb2), o,
                      ol);
    }
}

// The scan, scatter and order passes of an image in one launch, for bands of at
// most SORT_ATOMS atoms and SORT_CAP bins (launch latency bounds those passes
// there): a cluster of SORT_CL blocks per image, every block scanning the image's
// counts into its own shared memory (16 bits hold them), the atoms shared out over
// the blocks, one cluster barrier between the unordered slots and the order.  With
// more than SORT_BINS bins the scan goes by chunks and the starts are read back
// from memory.  Same slots as the five passes.
static_assert(SORT_ATOMS < 65536, "bin starts are kept in 16 bits");
template <typename T>
__device__ __forceinline__ void sort_image(const BandDev &b, int img, unsigned short *s_start,
                                           int *s_w) {
    using T4 = typename Vec4<T>::type;
    const ImgScalars &sc = b.sc[img];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    const int first = (int)(blockIdx.x % SORT_CL) * SORT_THREADS + tid;
    constexpr int STEP = SORT_CL * SORT_THREADS;
    const int n = b.n, nb = sc.nbins, nb1 = sc.nb[1], nb2 = sc.nb[2];
    const size_t base = (size_t)img * n;
    int *cnt = b.bin_count + (size_t)img * b.nbins_cap;
    int *start = b.bin_start + (size_t)img * (b.nbins_cap + 1);
    int before = 0;  // atoms of the chunks before
    for (int c = 0; c < nb; c += SORT_BINS) {
        const int m = min(SORT_BINS, nb - c);
        for (int k = tid; k < m; k += SORT_THREADS) s_start[k] = (unsigned short)cnt[c + k];
        __syncthreads();
        // an odd number of bins per thread spreads the threads over the banks
        const int per = ((m + SORT_THREADS - 1) / SORT_THREADS) | 1;
        const int k0 = min(tid * per, m), k1 = min(k0 + per, m);
        int sum = 0;
        for (int k = k0; k < k1; ++k) sum += s_start[k];
        int inc = sum;
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        if (lane == 31) s_w[w] = inc;
        __syncthreads();
        int run = before + inc - sum;
        for (int q = 0; q < SORT_THREADS / 32; ++q) {
            if (q < w) run += s_w[q];
            before += s_w[q];
        }
        for (int k = k0; k < k1; ++k) {
            const int v = s_start[k];
            s_start[k] = (unsigned short)run;
            run += v;
        }
        __syncthreads();
        for (int k = first; k < m; k += STEP) start[c + k] = s_start[k];
        if (c + m < nb) __syncthreads();  // the next chunk takes this one's place
    }
    if (first == 0) start[nb] = n;
    const bool held = nb <= SORT_BINS;  // uniform over the cluster
    if (!held) cluster_barrier();
    // what the cluster's other blocks wrote is read from L2
    const auto start_of = [&](int k) {
        return held ? (k < nb ? (int)s_start[k] : n) : __ldcg(start + k);
    };
    int *un = b.slot_unsorted + base;
    for (int i = first; i < n; i += STEP)
        un[start_of(b.atom_bin[base + i]) + b.atom_rank[base + i]] = i;
    cluster_barrier();
    // every block has read the counts: zero for the next build
    for (int k = first; k < nb; k += STEP) cnt[k] = 0;
    for (int i = first; i < n; i += STEP) {
        const int bin = b.atom_bin[base + i];
        const T4 o = ((const T4 *)b.atom_off)[base + i];
        const float4 ol = b.atom_off_lo[base + i];
        const int s0 = start_of(bin), s1 = start_of(bin + 1);
        int dst = s0;
        for (int q = s0; q < s1; ++q) dst += __ldcg(un + q) < i;
        order_atom<T>(b, base, i, dst, pack_bin(bin / (nb1 * nb2), (bin / nb2) % nb1, bin % nb2), o,
                      ol);
    }
}

template <typename T>
__global__ void __cluster_dims__(SORT_CL, 1, 1) __launch_bounds__(SORT_THREADS)
    k_bin_sort(const ImgRef *imgs, BandDev *bands) {
    __shared__ unsigned short s_start[SORT_BINS];
    __shared__ int s_w[SORT_THREADS / 32];
    const ImgRef r = imgs[blockIdx.x / SORT_CL];
    const BandDev b = bands[r.band];
    dep_sync();
    if (b.sc[r.img].rebuild) sort_image<T>(b, r.img, s_start, s_w);  // uniform over the cluster
}
// Sets of more images than SMs are shared out over a cluster per SM, which reads 32
// images' decisions at once: with a cluster per image, the blocks that find nothing
// to rebuild were a fifth of a step (256 bands of 31 atoms x 5 images, mixed: 168 us
// per step, 141 so; 64 bands of 256 to 28,000 atoms x 7 images: 1,545 us either way).
template <typename T>
__global__ void __cluster_dims__(SORT_CL, 1, 1) __launch_bounds__(SORT_THREADS)
    k_bin_sort_many(const ImgRef *imgs, int count, BandDev *bands) {
    __shared__ unsigned short s_start[SORT_BINS];
    __shared__ int s_w[SORT_THREADS / 32];
    const int clusters = gridDim.x / SORT_CL, step = 32 * clusters;
    const int l = (int)(threadIdx.x & 31) * clusters;
    dep_sync();
    // k: uniform over the cluster, as all that follows from it
    for (int k = blockIdx.x / SORT_CL; k < count; k += step) {
        const ImgRef f = imgs[min(k + l, count - 1)];
        unsigned todo =
            __ballot_sync(0xffffffffu, k + l < count && bands[f.band].sc[f.img].rebuild);
        for (; todo; todo &= todo - 1) {
            const ImgRef r = imgs[k + (__ffs(todo) - 1) * clusters];
            const BandDev b = bands[r.band];
            sort_image<T>(b, r.img, s_start, s_w);
            __syncthreads();  // the next image takes this one's place
        }
    }
}

// Cartesian positions R = R~ D (FP64) of a band's images (`per` blocks each), for
// output.
template <typename T>
__global__ void k_cartesian(BandDev *band, int per) {
    const ImgRef r = {0, (int)(blockIdx.x / per)};
    BandDev &b = *band;
    int i = (blockIdx.x % per) * blockDim.x + threadIdx.x;
    if (i >= b.n) return;
    const ImgScalars &sc = b.sc[r.img];
    const T *Xi = (const T *)b.X + ((size_t)r.img * b.rows + i) * 3;
    double x[3] = {(double)Xi[0], (double)Xi[1], (double)Xi[2]};
    double *o = b.cart + ((size_t)r.img * b.n + i) * 3;
    for (int c = 0; c < 3; ++c) o[c] = x[0] * sc.D[c] + x[1] * sc.D[3 + c] + x[2] * sc.D[6 + c];
}

// ---- launchers -------------------------------------------------------------

template <typename T>
void launch_mapback(const ImgRef *imgs, int count, BandDev *bands, int force, cudaStream_t s) {
    if (count <= 0) return;
    launch_dep(k_mapback<T>, count, 32, s, imgs, count, bands, force);
}
template <typename T>
void launch_bin_assign(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s,
                       cudaGraphConditionalHandle cond, int has_cond) {
    if (ntiles <= 0) return;
    launch_dep(k_bin_assign<T>, ntiles, TILE, s, tiles, bands, cond, has_cond);
}
void launch_bin_scan(const ImgRef *imgs, int count, int max_bins, BandDev *bands,
                     cudaStream_t s, int part) {
    if (count <= 0 || max_bins <= 0) return;
    dim3 grid(count, std::min((max_bins + SCAN_TILE - 1) / SCAN_TILE, 32));
    if (part == 0) launch_dep(k_bin_tilesum, grid, 256, s, imgs, bands);
    else if (part == 1) launch_dep(k_bin_tilescan, count, 1024, s, imgs, bands);
    else launch_dep(k_bin_scanfill, grid, 1024, s, imgs, bands);
}
void launch_bin_scatter(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s) {
    if (ntiles <= 0) return;
    launch_dep(k_bin_scatter, std::min(ntiles, gated_grid()), TILE, s, tiles, ntiles, bands);
}
template <typename T>
void launch_bin_order(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s) {
    if (ntiles <= 0) return;
    launch_dep(k_bin_order<T>, std::min(ntiles, gated_grid()), TILE, s, tiles, ntiles, bands);
}
template <typename T>
void launch_bin_sort(const ImgRef *imgs, int count, BandDev *bands, cudaStream_t s) {
    if (count <= 0) return;
    if (count <= sm_count())
        launch_dep(k_bin_sort<T>, count * SORT_CL, SORT_THREADS, s, imgs, bands);
    else
        launch_dep(k_bin_sort_many<T>, sm_count() * SORT_CL, SORT_THREADS, s, imgs, count, bands);
}
template <typename T>
void launch_cartesian(int N, int n, BandDev *band, cudaStream_t s) {
    if (N <= 0 || n <= 0) return;
    const int per = (n + 127) / 128;
    k_cartesian<T><<<N * per, 128, 0, s>>>(band, per);
}

#define CFNEB_INST(T)                                                                     \
    template void launch_mapback<T>(const ImgRef *, int, BandDev *, int, cudaStream_t);  \
    template void launch_bin_assign<T>(const Tile *, int, BandDev *, cudaStream_t,       \
                                       cudaGraphConditionalHandle, int);                 \
    template void launch_bin_order<T>(const Tile *, int, BandDev *, cudaStream_t);        \
    template void launch_bin_sort<T>(const ImgRef *, int, BandDev *, cudaStream_t);       \
    template void launch_cartesian<T>(int, int, BandDev *, cudaStream_t);
CFNEB_INST(float)
CFNEB_INST(double)
#undef CFNEB_INST

}  // namespace cfneb
