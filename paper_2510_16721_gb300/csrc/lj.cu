// Lennard-Jones energy, forces and virial over the cell list.
//
// phi(r) = 4 eps [(sigma/r)^12 - (sigma/r)^6] - phi(rc) (energy shifted when
// requested); U_i = 1/2 sum_j phi(r_ij) (the per-atom split of Sec. II.B,
// Eq. U).  For a pair potential the force on i due to j of the
// derivation of Eq. V2, f^ij = dU_i/dr^ij - dU_j/dr^ji, is phi'(r) r^ij / r,
// so F_i = sum_j phi'(r) r^ij / r and V = -1/2 sum_ij r^ij (x) f^ij.
//
// Atoms are taken in cell-list slot order (neighbouring threads share
// neighbour bins, so their loads hit L1), one thread per atom or, in bands too
// small to fill the chip that way, 2..32 lanes per atom (BandDev::tile).  Full
// neighbour enumeration (every pair visited from both ends): no atomics, fixed
// summation order.  Arithmetic in T (float on the mixed path) with T
// per-atom accumulators; tile energies and virials are summed in FP64.  The
// epilogue applies the cell filter's atom-row transform F D^T (Sec. II.C).
#include "common.cuh"

namespace cfneb {

// sigma^2 / r^2: FP32 by the fast division intrinsic (2 ulp: ~1e-6 of a
// pair force, far inside the mixed path's 1e-4 force tolerance), FP64 by
// Newton steps (~1 ulp; a divide is a long chain of FP64 instructions)
__device__ inline float lj_sr2(float sig2, float r2) { return __fdividef(sig2, r2); }
__device__ inline double lj_sr2(double sig2, double r2) { return sig2 * rcp64_pos(r2); }

// r2 < rc2 and r2 > 0 for a squared distance (never negative)
__device__ inline bool lj_inside(float r2, float rc2) { return r2 < rc2 && r2 > 0.0f; }
__device__ inline bool lj_inside(double r2, double rc2) {
    return less_pos(r2, rc2) && __double_as_longlong(r2) != 0;
}

// Per-thread LJ accumulators: force on atom i, energy sum, virial, pair count.
// FP64 keeps force and virial in units of c24 = 24 eps / sigma^2 and scales
// once per atom: two FP64 instructions less per pair.  FP32 scales each pair:
// its steps feed relaxations that amplify a changed rounding, for no gain (the
// list kernel waits on its gathers).
template <typename T>
struct LJAcc {
    T fx = 0, fy = 0, fz = 0, e = 0;
    T v00 = 0, v01 = 0, v02 = 0, v11 = 0, v12 = 0, v22 = 0;
    int cnt = 0;
    // pair vector (rx, ry, rz) with |r|^2 = r2
    __device__ inline void pair(T rx, T ry, T rz, T r2, T sig2, T c24) {
        const T sr2 = lj_sr2(sig2, r2);
        const T sr6 = sr2 * sr2 * sr2;
        // phi'(r)/r = 24 eps (sr6 - 2 sr6^2) / r^2
        T fr;
        if constexpr (sizeof(T) == 4) {
            fr = c24 * sr2 * sr6 * ((T)1 - (T)2 * sr6);
            e += sr6 * (sr6 - (T)1);
        } else {
            const T sr12 = sr6 * sr6;
            fr = fma((T)-2, sr12, sr6) * sr2;
            e += sr12 - sr6;
        }
        const T frx = fr * rx, fry = fr * ry, frz = fr * rz;
        fx += frx;
        fy += fry;
        fz += frz;
        v00 += frx * rx;
        v01 += frx * ry;
        v02 += frx * rz;
        v11 += fry * ry;
        v12 += fry * rz;
        v22 += frz * rz;
        ++cnt;
    }
};

// floor(a / b) for b > 0
__device__ inline int floor_div(int a, int b) { return a >= 0 ? a / b : -((b - 1 - a) / b); }

// Code of a (bin offset d, periodic wrap t) combination along one axis.  For
// any bin of an axis of nb bins, t is floor(d / nb) or floor(d / nb) + 1, so
// 2 (d + m) + (t - floor(d / nb)) < 2 (2m + 1) <= 30 identifies it.
__device__ inline int axis_code(int d, int t, int m, int nb) {
    // no division where the stencil is narrower than the axis
    return 2 * (d + m) + (t - (nb > m ? d >> 31 : floor_div(d, nb)));
}

// Which of the two ends of a pair of an atom with its own periodic image a
// code is: along the first axis with a non-zero displacement in whole lattice
// vectors the two ends have opposite signs; true for the negative one.
__device__ inline bool lj_back(uint32_t code, const int *m, const int *nb) {
    for (int a = 0; a < 3; ++a) {
        const int i = (code >> (5 * a)) & 31u, d = (i >> 1) - m[a];
        const int t = floor_div(d, nb[a]) + (i & 1);
        if (t) return t < 0;
    }
    return false;
}

// Neighbour-list entry: slot in bits 0-16, i0 + LJ_AXIS i1 in bits 17-26 and
// i2 in bits 27-31 (i_a the axis codes).  The list path therefore needs
// n <= 2^17 atoms per image.
constexpr int LJ_AXIS = 30;
// entries the list force kernel takes per iteration (lists are padded to it)
constexpr int LJ_UNROLL = 4;
__device__ inline uint32_t lj_entry(int q, int i01, int i2) {
    return (uint32_t)q | ((uint32_t)i01 << 17) | ((uint32_t)i2 << 27);
}

// Bins farther than the list cutoff and a bin's half diagonal from the atom hold
// no candidate.  Of the 125 half-cutoff bins of a stencil about a third are: a row
// is walked over the part of it inside that sphere (ibb = 1 / |b|^2 of the innermost
// bin vector b).  24 bands' lists 183 -> 169 us, the FP32 walk of 62,500 atoms
// 124.5 -> 115.3 us.
struct LJTrim {
    float r2, ibb;
};

// Visits every cell-list candidate of the atom with FP32 offset oi in bin
// (b0, b1, b2) along the stencil row (d0, d1): visit(q, ux, uy, uz, i0, i1,
// i2) with (ux, uy, uz) the FP32 pair vector to slot q and i0, i1, i2 the axis
// codes of its (offset, wrap).  Where the row, along the innermost bin axis,
// does not wrap around the cell its bins are consecutive in the cell list,
// so it is one contiguous range of atoms (one pair of bin-start loads
// instead of one per bin) and each atom's displacement comes from its own
// innermost bin index, stored in the offset's fourth lane.  Rows that wrap
// are walked bin by bin.  AHEAD: the next candidate is loaded under the
// current one's work (worth its registers where few warps are resident).
template <bool AHEAD, typename Visit>
__device__ inline void lj_row(const float4 *off, const int *start, const float4 &oi, int b0, int b1,
                              int b2, int d0, int d1, const float *s_bv, const float *s_dh,
                              const int *s_nb, const int *s_m, const LJTrim &trim,
                              Visit &&visit) {
    const int nb0 = s_nb[0], nb1 = s_nb[1], nb2 = s_nb[2];
    const int m0 = s_m[0], m1 = s_m[1], m2 = s_m[2];
    const bool row_ok = (b2 - m2 >= 0) && (b2 + m2 < nb2);
    int w0 = b0 + d0, t0 = 0;
    while (w0 < 0) { w0 += nb0; --t0; }
    while (w0 >= nb0) { w0 -= nb0; ++t0; }
    int w1 = b1 + d1, t1 = 0;
    while (w1 < 0) { w1 += nb1; --t1; }
    while (w1 >= nb1) { w1 -= nb1; ++t1; }
    const int i0 = axis_code(d0, t0, m0, nb0), i1 = axis_code(d1, t1, m1, nb1);
    const int rowbase = (w0 * nb1 + w1) * nb2;
    // displacement for d2 = 0 (row base) and the wrap remainder
    const float cx = (d0 * s_bv[0] + d1 * s_bv[3]) + (t0 * s_dh[0] + t1 * s_dh[3]);
    const float cy = (d0 * s_bv[1] + d1 * s_bv[4]) + (t0 * s_dh[1] + t1 * s_dh[4]);
    const float cz = (d0 * s_bv[2] + d1 * s_bv[5]) + (t0 * s_dh[2] + t1 * s_dh[5]);
    const float px = cx - oi.x, py = cy - oi.y, pz = cz - oi.z;  // to the bin at d2 = 0
    if (row_ok) {
        // |p + d2 b|^2 <= R^2, in units of |b|: fourth powers of a length in metres
        // would leave FP32's range
        const float pb = (px * s_bv[6] + py * s_bv[7] + pz * s_bv[8]) * trim.ibb;
        const float disc = pb * pb - (px * px + py * py + pz * pz - trim.r2) * trim.ibb;
        if (!(disc >= 0.0f)) return;
        float h;  // an estimate: R has a margin of 0.1%
        asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(h) : "f"(disc));
        const int lo = max(-m2, (int)ceilf(-pb - h));
        const int hi = min(m2, (int)floorf(h - pb));
        if (lo > hi) return;
        const int q0 = start[rowbase + b2 + lo], q1 = start[rowbase + b2 + hi + 1];
        float4 next;
        if (AHEAD && q0 < q1) next = off[q0];
        for (int q = q0; q < q1; ++q) {
            const float4 oj = AHEAD ? next : off[q];
            if (AHEAD && q + 1 < q1) next = off[q + 1];
            const float d2 = oj.w - (float)b2;
            const float ex = cx + d2 * s_bv[6], ey = cy + d2 * s_bv[7], ez = cz + d2 * s_bv[8];
            // no wrap along the row: t2 = 0, and |d2| <= m2 < nb2
            const int id2 = (int)d2;
            visit(q, (oj.x - oi.x) + ex, (oj.y - oi.y) + ey, (oj.z - oi.z) + ez, i0, i1,
                  2 * (id2 + m2) + (id2 < 0 ? 1 : 0));
        }
    } else {
        for (int d2 = -m2; d2 <= m2; ++d2) {
            int w2 = b2 + d2, t2 = 0;
            while (w2 < 0) { w2 += nb2; --t2; }
            while (w2 >= nb2) { w2 -= nb2; ++t2; }
            const int i2 = axis_code(d2, t2, m2, nb2);
            const float ex = cx + (d2 * s_bv[6] + t2 * s_dh[6]);
            const float ey = cy + (d2 * s_bv[7] + t2 * s_dh[7]);
            const float ez = cz + (d2 * s_bv[8] + t2 * s_dh[8]);
            const float dx = ex - oi.x, dy = ey - oi.y, dz = ez - oi.z;
            if (dx * dx + dy * dy + dz * dz > trim.r2) continue;
            const int q1 = start[rowbase + w2 + 1];
            for (int q = start[rowbase + w2]; q < q1; ++q) {
                const float4 oj = off[q];
                visit(q, (oj.x - oi.x) + ex, (oj.y - oi.y) + ey, (oj.z - oi.z) + ez, i0, i1, i2);
            }
        }
    }
}

// A lane's rows of the stencil: lane, lane + lanes, ... of the (2 m0 + 1)(2 m1
// + 1) rows, as (d0, d1) stepped without a division per row.
struct LJRows {
    int d0, d1, m0, m1;
    __device__ LJRows(const int *m, int lane) : d0(-m[0]), d1(-m[1]), m0(m[0]), m1(m[1]) {
        step(lane);
    }
    __device__ bool more() const { return d0 <= m0; }
    __device__ void step(int k) {
        d1 += k;
        while (d1 > m1) {
            d1 -= 2 * m1 + 1;
            ++d0;
        }
    }
};

// Per-block staging of an image's bin geometry and the LJ constants in T
template <typename T>
struct LJGeom {
    T bv[9], dh[9], D[9];
    T rc2, sig2, c24, e4, ephi;   // rc^2, sigma^2, 24 eps / sigma^2, 4 eps, phi(rc)
    float screen;                 // squared screen radius of the walk, with a margin
    float bvf[9], dhf[9];         // bin vectors and wrap terms in FP32 (the walk)
    int nb[3], m[3];
    LJTrim trim;                  // which part of a row can hold a candidate
};
template <typename T>
__device__ inline void lj_stage(LJGeom<T> &g, const ImgScalars &sc, const BandParams &bp,
                                bool fp64_band, bool list) {
    if (threadIdx.x == 0) {
        const LJParams p = *(const LJParams *)bp.pot;
        g.rc2 = (T)p.rc2;
        g.sig2 = (T)p.sig2;
        g.c24 = (T)p.c24;
        g.e4 = (T)p.e4;
        g.ephi = (T)p.ephi_c;
        // lists cover rl; a walk that evaluates its candidates is cut at rc
        // (the test in T decides: the margin only has to cover the screen's
        // FP32 rounding)
        if (list) g.screen = fp64_band ? screen_r2<double>(bp.rl, sc) : screen_r2<float>(bp.rl, sc);
        else g.screen = fp64_band ? screen_r2<double>(p.rc, sc) : (float)p.rc2 * 1.001f;
    }
    if (threadIdx.x == 32) {
        // a bin's corners lie within rho of its centre, and so its atoms at the
        // build; kept bins are walked with atoms that have moved by up to the skin
        const float *v = sc.bvf;
        float rho2 = 0.0f;
        for (int k = 0; k < 4; ++k) {
            float q = 0.0f;
            for (int c = 0; c < 3; ++c) {
                const float x =
                    v[c] + (k & 1 ? v[3 + c] : -v[3 + c]) + (k & 2 ? v[6 + c] : -v[6 + c]);
                q += 0.25f * x * x;
            }
            rho2 = fmaxf(rho2, q);
        }
        const float rl = (float)(bp.rl > 0.0 ? bp.rl : bp.rc);
        const float R = 1.001f * (rl + sqrtf(rho2) + (list ? 0.0f : (float)bp.skin));
        g.trim.r2 = R * R;
        g.trim.ibb = 1.0f / (v[6] * v[6] + v[7] * v[7] + v[8] * v[8]);
    }
    if (threadIdx.x < 9) {
        g.bv[threadIdx.x] = (T)sc.bv[threadIdx.x];
        g.dh[threadIdx.x] = (T)sc.dh[threadIdx.x];
        g.D[threadIdx.x] = (T)sc.D[threadIdx.x];
        g.bvf[threadIdx.x] = sc.bvf[threadIdx.x];
        g.dhf[threadIdx.x] = sc.dhf[threadIdx.x];
    }
    if (threadIdx.x < 3) {
        g.nb[threadIdx.x] = sc.nb[threadIdx.x];
        g.m[threadIdx.x] = sc.m[threadIdx.x];
    }
}

// Writes the generalised atom force F D^T of slot t (row vector times D^T)
// and the tile's energy, virial and pair-count partials.
template <typename T>
__device__ inline void lj_finish(const LJAcc<T> &A, const LJGeom<T> &g, const BandDev &b,
                                 const Tile &tl, int t, bool active) {
    const T scale = sizeof(T) == 4 ? (T)1 : g.c24;
    if (active) {
        const T fx = scale * A.fx, fy = scale * A.fy, fz = scale * A.fz;
        const T g0 = fx * g.D[0] + fy * g.D[1] + fz * g.D[2];
        const T g1 = fx * g.D[3] + fy * g.D[4] + fz * g.D[5];
        const T g2 = fx * g.D[6] + fy * g.D[7] + fz * g.D[8];
        const int atom = b.slot_atom[(size_t)tl.img * b.n + t];
        T *F = (T *)b.F + ((size_t)tl.img * b.rows + atom) * 3;
        F[0] = g0;
        F[1] = g1;
        F[2] = g2;
    }
    // U_i = 1/2 sum_j [4 eps (sr12 - sr6) - phi(rc)];  V = -1/2 sum r (x) f,
    // written as the symmetric virial in row-major order
    const T vs = (T)(-0.5) * scale;
    T acc[12];
    acc[0] = (T)0.5 * (g.e4 * A.e - g.ephi * (T)A.cnt);
    acc[1] = vs * A.v00;
    acc[2] = acc[4] = vs * A.v01;
    acc[3] = acc[7] = vs * A.v02;
    acc[5] = vs * A.v11;
    acc[6] = acc[8] = vs * A.v12;
    acc[9] = vs * A.v22;
    acc[10] = (T)A.cnt;
    acc[11] = (T)0;
    double *part = b.atom_part + ((size_t)tl.img * b.atpi + tl.t) * NPART;
    if (sizeof(T) == 4) block_sum_store<12, T>(acc, part);
    else block_sum_store_tr<12, T>(acc, part);  // 17 FP64 additions per warp instead of 60
}

// Sums v over the `lanes` (a power of two) adjacent lanes that share an atom.
template <typename T>
__device__ inline T lane_group_sum(T v, int lanes) {
    for (int o = 1; o < lanes; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Direct path (bands without a neighbour list: no skin, or more atoms per
// image than a list entry can index).  The stencil's rows are dealt to the
// lanes of the atom.
//
// FP32 evaluates a candidate where the walk finds it (62,500 atoms: 205 us with
// one lane per atom, latency-bound; 196 us with four, issue-bound).
//
// FP64 is bound by its pipe: the walk sees ~370-500 candidates per atom for
// ~78 pairs inside rc, and in a warp nearly every candidate is inside for some
// lane, so a pair term evaluated where it is found costs the warp its ~40 FP64
// instructions (~64 cycles each) that many times: 1116 us for 19,380 atoms,
// and 2093 us for the FP64 energies of 62,500.  There the walk runs in FP32 on
// the rounded offsets and each thread keeps the candidates inside the screen
// in shared memory; between rows, when some lane of the warp has little room
// left, and at the end, groups of lanes share out what they kept evenly and
// evaluate it, every lane busy (now 165 us, 99 us of it the FP64 pipe's, and
// 202 us).
//
// A kept candidate is one word (slot in 17 bits, three axis codes of 5) where
// the image has at most 2^17 atoms, else two.  Rows of LJ_KEEP words per
// thread, an odd stride apart (a group reads consecutive words of one row,
// threads append to their own).
constexpr int LJ_KEEP = 56, LJ_KEEP_STRIDE = LJ_KEEP + 1;
constexpr int LJ_ROOM = 16;      // a flush leaves room for this many words per row
struct LJKept {
    uint32_t word[TILE * LJ_KEEP_STRIDE];
    int cnt[TILE];
};

// Evaluates what the threads of each group of `group` adjacent lanes kept:
// term(q, code, column) in the same order whatever the kernel's schedule, item
// i of the group's concatenated rows on its lane i mod group.
template <typename Term>
__device__ inline void lj_share(LJKept &kp, int group, bool wide, int &kept, Term &&term) {
    const int tid = threadIdx.x, lane = tid & (group - 1), g0 = tid - lane;
    kp.cnt[tid] = kept;
    __syncwarp();
    int total = kept;
    for (int o = 1; o < group; o <<= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    int col = g0, k = lane;
    for (int i = lane; i < total; i += group, k += group) {
        while (k >= kp.cnt[col]) k -= kp.cnt[col++];
        const uint32_t *w = kp.word + col * LJ_KEEP_STRIDE + (wide ? 2 * k : k);
        if (wide) term((int)w[0], w[1], col);
        else term((int)(w[0] & 0x1FFFFu), w[0] >> 17, col);
    }
    __syncwarp();
    kept = 0;
}

// Walks the stencil of slot t (this thread's share of its rows) and keeps the
// candidates inside g.screen; HALF: only one of each pair's two ends.
template <typename TS, bool HALF, typename T, typename Term>  // TS: the band's storage type
__device__ inline void lj_walk_keep(const BandDev &b, const Tile &tl, const LJGeom<T> &g,
                                    LJKept &kp, int group, int t, int lane, int lanes,
                                    Term &&term) {
    const int n = b.n, tid = threadIdx.x;
    const bool wide = n > LJ_LIST_MAX_ATOMS, active = t < n;
    const int cap = wide ? LJ_KEEP / 2 : LJ_KEEP, room = wide ? LJ_ROOM / 2 : LJ_ROOM;
    const size_t base = (size_t)tl.img * n;
    const float4 *off = screen_off<TS>(b, base);
    const int *start = b.bin_start + (size_t)tl.img * (b.nbins_cap + 1);
    int b0 = 0, b1 = 0, b2 = 0;
    float4 oi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (active) {
        unpack_bin(b.slot_bin[base + t], b0, b1, b2);
        oi = off[t];
    }
    // the code of zero offset and wrap (the atom itself)
    const uint32_t zero = (uint32_t)(2 * g.m[0] | (2 * g.m[1] << 5) | (2 * g.m[2] << 10));
    uint32_t *row = kp.word + tid * LJ_KEEP_STRIDE;
    int kept = 0;
    LJRows r(g.m, lane);
    const int rows = (2 * g.m[0] + 1) * (2 * g.m[1] + 1);
    for (int r0 = 0; r0 < rows; r0 += lanes, r.step(lanes)) {  // uniform over the block
        if (active && r.more())
            lj_row<true>(
                off, start, oi, b0, b1, b2, r.d0, r.d1, g.bvf, g.dhf, g.nb, g.m, g.trim,
                [&](int q, float ux, float uy, float uz, int i0, int i1, int i2) {
                    if (!(ux * ux + uy * uy + uz * uz < g.screen)) return;
                    if (HALF && q < t) return;
                    const uint32_t code = (uint32_t)(i0 | (i1 << 5) | (i2 << 10));
                    if (q == t && (code == zero || (HALF && lj_back(code, g.m, g.nb)))) return;
                    if (kept == cap) {  // a very dense row: this thread alone
                        for (int k = 0; k < kept; ++k) {
                            if (wide) term((int)row[2 * k], row[2 * k + 1], tid);
                            else term((int)(row[k] & 0x1FFFFu), row[k] >> 17, tid);
                        }
                        kept = 0;
                    }
                    if (wide) {
                        row[2 * kept] = (uint32_t)q;
                        row[2 * kept + 1] = code;
                    } else {
                        row[kept] = (uint32_t)q | (code << 17);
                    }
                    ++kept;
                });
        if (__any_sync(0xffffffffu, kept > cap - room)) lj_share(kp, group, wide, kept, term);
    }
    lj_share(kp, group, wide, kept, term);
}

// FP64 displacements of the axis codes, d bv + t dh: of the first two axes
// together (a table of LJ_C01 pairs; wider stencils add the two), and of the
// innermost one.  Staged by the block.
constexpr int LJ_C01 = 400;
struct LJDisp {
    double c01[LJ_C01 * 3], a[2][32][3], c2[32][3];
    int l0, l1;   // codes per axis; l0 l1 <= LJ_C01: the table is used
};
__device__ inline void lj_disp_stage(LJDisp &D, const LJGeom<double> &g) {
    for (int k = threadIdx.x; k < 96; k += TILE) {
        const int a = k / 32, i = k % 32;
        const int d = (i >> 1) - g.m[a];
        const int t = floor_div(d, g.nb[a]) + (i & 1);
        for (int c = 0; c < 3; ++c) {
            const double v = (double)d * g.bv[3 * a + c] + (double)t * g.dh[3 * a + c];
            if (a < 2) D.a[a][i][c] = v;
            else D.c2[i][c] = v;
        }
    }
    const int l0 = 2 * (2 * g.m[0] + 1), l1 = 2 * (2 * g.m[1] + 1);
    if (threadIdx.x == 0) {
        D.l0 = l0;
        D.l1 = l1;
    }
    __syncthreads();
    if (l0 * l1 <= LJ_C01)
        for (int k = threadIdx.x; k < l0 * l1 * 3; k += TILE)
            D.c01[k] = D.a[0][(k / 3) % l0][k % 3] + D.a[1][k / 3 / l0][k % 3];
}
__device__ inline void lj_disp(const LJDisp &D, uint32_t code, double &x, double &y, double &z) {
    const int i0 = code & 31u, i1 = (code >> 5) & 31u, i2 = (code >> 10) & 31u;
    const double *c2 = D.c2[i2];
    if (D.l0 * D.l1 <= LJ_C01) {
        const double *c = D.c01 + 3 * (i0 + D.l0 * i1);
        x += c[0] + c2[0];
        y += c[1] + c2[1];
        z += c[2] + c2[2];
    } else {
        const double *c = D.a[0][i0], *d = D.a[1][i1];
        x += c[0] + d[0] + c2[0];
        y += c[1] + d[1] + c2[1];
        z += c[2] + d[2] + c2[2];
    }
}

template <typename T> __global__ void k_lj(const Tile *tiles, BandDev *bands);
template <>
__global__ void __launch_bounds__(TILE, 8) k_lj<float>(const Tile *tiles, BandDev *bands) {
    dep_sync();
    Tile tl = tiles[blockIdx.x];
    BandDev &b = bands[tl.band];
    if (b.lj_cap > 0) return;  // uniform over the block: the list path runs
    const ImgScalars &sc = b.sc[tl.img];
    __shared__ LJGeom<float> g;
    lj_stage(g, sc, *b.bp, false, false);
    __syncthreads();
    const int n = b.n, lanes = TILE / b.tile, lane = threadIdx.x % lanes;
    const int t = tl.t * b.tile + (int)threadIdx.x / lanes;
    const size_t base = (size_t)tl.img * n;
    const float4 *off = (const float4 *)b.slot_off + base;
    const int *start = b.bin_start + (size_t)tl.img * (b.nbins_cap + 1);
    const float rc2 = g.rc2, sig2 = g.sig2, c24 = g.c24;
    LJAcc<float> A;
    if (t < n) {
        int b0, b1, b2;
        unpack_bin(b.slot_bin[base + t], b0, b1, b2);
        const float4 oi = off[t];
        for (LJRows r(g.m, lane); r.more(); r.step(lanes))
            lj_row<false>(off, start, oi, b0, b1, b2, r.d0, r.d1, g.bvf, g.dhf, g.nb, g.m, g.trim,
                          [&](int, float ux, float uy, float uz, int, int, int) {
                              const float r2 = ux * ux + uy * uy + uz * uz;
                              // r2 == 0 only for the atom itself at zero shift
                              if (lj_inside(r2, rc2)) A.pair(ux, uy, uz, r2, sig2, c24);
                          });
    }
    A.fx = lane_group_sum(A.fx, lanes);
    A.fy = lane_group_sum(A.fy, lanes);
    A.fz = lane_group_sum(A.fz, lanes);
    lj_finish(A, g, b, tl, t, t < n && lane == 0);
}

template <>
__global__ void __launch_bounds__(TILE) k_lj<double>(const Tile *tiles, BandDev *bands) {
    dep_sync();
    using T4 = typename Vec4<double>::type;
    Tile tl = tiles[blockIdx.x];
    BandDev &b = bands[tl.band];
    if (b.lj_cap > 0) return;  // uniform over the block: the list path runs
    const ImgScalars &sc = b.sc[tl.img];
    __shared__ LJGeom<double> g;
    __shared__ LJDisp D;
    __shared__ LJKept kp;
    lj_stage(g, sc, *b.bp, true, false);
    __syncthreads();
    lj_disp_stage(D, g);
    __syncthreads();
    const int n = b.n, lanes = TILE / b.tile, lane = threadIdx.x % lanes;
    const int t = tl.t * b.tile + (int)threadIdx.x / lanes;
    const T4 *off = (const T4 *)b.slot_off + (size_t)tl.img * n;
    const double rc2 = g.rc2, sig2 = g.sig2, c24 = g.c24;
    T4 oi = {};
    if (t < n) oi = off[t];
    LJAcc<double> A;
    lj_walk_keep<double, false>(b, tl, g, kp, lanes, t, lane, lanes,
                                [&](int q, uint32_t code, int) {
                                    const T4 oj = off[q];
                                    double x = oj.x - oi.x, y = oj.y - oi.y, z = oj.z - oi.z;
                                    lj_disp(D, code, x, y, z);
                                    const double r2 = x * x + y * y + z * z;
                                    if (lj_inside(r2, rc2)) A.pair(x, y, z, r2, sig2, c24);
                                });
    A.fx = lane_group_sum(A.fx, lanes);
    A.fy = lane_group_sum(A.fy, lanes);
    A.fz = lane_group_sum(A.fz, lanes);
    lj_finish(A, g, b, tl, t, t < n && lane == 0);
}

// FP64 energies of an LJ band (reported paths, single points), from the cell
// list like k_lj<double>: FP32 walk, kept candidates shared out over the whole
// warp.  Each pair is taken at one of its ends only (half the FP64 work: a
// total needs no per-atom split).  FP32 bands form the pair vector from
// two-term offsets: the leading difference as an exact FP32 sum (two-sum), so
// that FP64 starts at two additions per component instead of four conversions
// and three additions.
template <typename T> struct LJEnd;  // an atom's offset in shared memory
template <> struct LJEnd<float> { float4 o, l; };
template <> struct LJEnd<double> { double x, y, z; };
__device__ inline double lj_diff64(float oj, float ojl, float oi, float oil) {
    const float s = __fsub_rn(oj, oi), bb = __fsub_rn(s, oj);
    const float e = __fsub_rn(__fsub_rn(oj, __fsub_rn(s, bb)), __fadd_rn(oi, bb));
    return f2d(s) + f2d(__fadd_rn(__fsub_rn(ojl, oil), e));
}
__device__ inline void lj_delta(const float4 &o, const float4 &l, const LJEnd<float> &i, double &x,
                                double &y, double &z) {
    x = lj_diff64(o.x, l.x, i.o.x, i.l.x);
    y = lj_diff64(o.y, l.y, i.o.y, i.l.y);
    z = lj_diff64(o.z, l.z, i.o.z, i.l.z);
}

template <typename T>
__global__ void __launch_bounds__(TILE) k_lj_energy64(const Tile *tiles, BandDev *bands) {
    using T4 = typename Vec4<T>::type;
    Tile tl = tiles[blockIdx.x];
    BandDev &b = bands[tl.band];
    const ImgScalars &sc = b.sc[tl.img];
    __shared__ LJGeom<double> g;
    __shared__ LJDisp D;
    __shared__ LJKept kp;
    __shared__ LJEnd<T> s_end[TILE];
    lj_stage(g, sc, *b.bp, sizeof(T) == 8, false);
    __syncthreads();
    lj_disp_stage(D, g);
    const int n = b.n, lanes = TILE / b.tile, lane = threadIdx.x % lanes;
    const int t = tl.t * b.tile + (int)threadIdx.x / lanes;
    const T4 *off = (const T4 *)b.slot_off + (size_t)tl.img * n;
    const float4 *offl = b.slot_off_lo + (size_t)tl.img * n;
    if (t < n && lane == 0) {
        LJEnd<T> &s = s_end[threadIdx.x / lanes];
        const T4 o = off[t];
        if constexpr (sizeof(T) == 4) s = {o, offl[t]};
        else s = {o.x, o.y, o.z};
    }
    __syncthreads();
    const double rc2 = g.rc2, sig2 = g.sig2;
    double e = 0.0;
    int cnt = 0;
    lj_walk_keep<T, true>(b, tl, g, kp, 32, t, lane, lanes, [&](int q, uint32_t code, int col) {
        const LJEnd<T> &i = s_end[col / lanes];
        const T4 oj = off[q];
        double x, y, z;
        if constexpr (sizeof(T) == 4) {
            lj_delta(oj, offl[q], i, x, y, z);
        } else {
            x = oj.x - i.x;
            y = oj.y - i.y;
            z = oj.z - i.z;
        }
        lj_disp(D, code, x, y, z);
        const double r2 = x * x + y * y + z * z;
        if (lj_inside(r2, rc2)) {
            const double sr2 = sig2 * rcp64_pos(r2), sr6 = sr2 * sr2 * sr2;
            e += fma(sr6, sr6, -sr6);
            ++cnt;
        }
    });
    double acc[1] = {g.e4 * e - g.ephi * (double)cnt}, tot[1];
    block_sum<1>(acc, tot);
    if (threadIdx.x == 0) b.atom_part[((size_t)tl.img * b.atpi + tl.t) * NPART] = tot[0];
}

// Neighbour list of a rebuilt image (bands with a skin): one thread per atom (or
// several lanes, lj_list_lanes) walks the cell-list stencil and keeps every candidate
// within rl, coalesced as [entry][atom].  Entries inside rc at the build come first and those of
// the skin shell after them, so that the force kernel's warps mostly agree
// on which entries have a pair term.  Images that keep their cell list keep
// their list too.  The walk runs in FP32 in both precisions: FP64 bands
// screen on their rounded offsets (entries are tested again in FP64 by the
// force kernel).
template <typename T>
__device__ inline void lj_list_atom(const BandDev &b, const Tile &tl, const LJGeom<float> &g,
                                    int t) {
    const int n = b.n, cap = b.lj_cap;
    const size_t base = (size_t)tl.img * n;
    const float4 *off = screen_off<T>(b, base);
    const int *start = b.bin_start + (size_t)tl.img * (b.nbins_cap + 1);
    uint32_t *L = (uint32_t *)b.nbr_slot + (size_t)tl.img * cap * n + t;
    const float rc2 = g.rc2, screen = g.screen;
    // the atom itself: slot t at zero offset and wrap
    const uint32_t self =
        lj_entry(t, 2 * g.m[0] + LJ_AXIS * 2 * g.m[1], 2 * g.m[2]);
    int nin = 0, nsh = 0;
    const float4 oi = off[t];
    int b0, b1, b2;
    unpack_bin(b.slot_bin[base + t], b0, b1, b2);
    for (int d0 = -g.m[0]; d0 <= g.m[0]; ++d0)
        for (int d1 = -g.m[1]; d1 <= g.m[1]; ++d1)
            lj_row<false>(off, start, oi, b0, b1, b2, d0, d1, g.bvf, g.dhf, g.nb, g.m, g.trim,
                          [&](int q, float ux, float uy, float uz, int i0, int i1, int i2) {
                              const float r2 = ux * ux + uy * uy + uz * uz;
                              if (!(r2 < screen)) return;
                              const uint32_t e = lj_entry(q, i0 + LJ_AXIS * i1, i2);
                              if (e == self) return;
                              if (nin + nsh < cap)
                                  L[(size_t)(r2 < rc2 ? nin : cap - 1 - nsh) * n] = e;
                              if (r2 < rc2) ++nin;
                              else ++nsh;
                          });
    const int total = nin + nsh;
    if (total > cap) {
        // not every slot of [0, cap) holds an entry: none is read
        atomicOr(&b.bp->status, ST_NBR_OVERFLOW);
        b.nbr_cnt[base + t] = 0;
        return;
    }
    // the shell block [cap - nsh, cap) moves down behind the inner entries,
    // and the atom itself pads the list to a whole number of LJ_UNROLL
    // entries (cap is a multiple of 8; the pair term skips r = 0)
    for (int k = 0; k < nsh; ++k) L[(size_t)(nin + k) * n] = L[(size_t)(cap - nsh + k) * n];
    const int padded = (total + LJ_UNROLL - 1) / LJ_UNROLL * LJ_UNROLL;
    for (int k = total; k < padded; ++k) L[(size_t)k * n] = self;
    b.nbr_cnt[base + t] = padded;
}

// The same list by the `lanes` lanes of an atom (bands whose tiles hold fewer
// atoms than threads): each walks a share of the stencil's rows, once to count its
// entries and once to store them where the counts of the lanes before it put them.
// Whole warps call this (t >= n: no atom).  FP64 steps that rebuild, one thread per
// atom -> lanes: 31 atoms 55.2 -> 49.7 us, 2,915 atoms x 5 images 207 -> 175 us.
template <typename T>
__device__ inline void lj_list_lanes(const BandDev &b, const Tile &tl, const LJGeom<float> &g,
                                     int t, int lane, int lanes) {
    const int n = b.n, cap = b.lj_cap;
    const size_t base = (size_t)tl.img * n;
    const float4 *off = screen_off<T>(b, base);
    const int *start = b.bin_start + (size_t)tl.img * (b.nbins_cap + 1);
    uint32_t *L = (uint32_t *)b.nbr_slot + (size_t)tl.img * cap * n + t;
    const float rc2 = g.rc2, screen = g.screen;
    const uint32_t self = lj_entry(t, 2 * g.m[0] + LJ_AXIS * 2 * g.m[1], 2 * g.m[2]);
    const int w1 = 2 * g.m[1] + 1, rows = (2 * g.m[0] + 1) * w1;
    const int r0 = t < n ? rows * lane / lanes : 0, r1 = t < n ? rows * (lane + 1) / lanes : 0;
    float4 oi = make_float4(0, 0, 0, 0);
    int b0 = 0, b1 = 0, b2 = 0;
    if (t < n) {
        oi = off[t];
        unpack_bin(b.slot_bin[base + t], b0, b1, b2);
    }
    const auto walk = [&](auto keep) {
        for (int r = r0; r < r1; ++r)
            lj_row<false>(off, start, oi, b0, b1, b2, r / w1 - g.m[0], r % w1 - g.m[1], g.bvf,
                          g.dhf, g.nb, g.m, g.trim,
                          [&](int q, float ux, float uy, float uz, int i0, int i1, int i2) {
                              const float r2 = ux * ux + uy * uy + uz * uz;
                              if (!(r2 < screen)) return;
                              const uint32_t e = lj_entry(q, i0 + LJ_AXIS * i1, i2);
                              if (e != self) keep(e, r2 < rc2);
                          });
    };
    int nin = 0, nsh = 0, tin, tsh;
    walk([&](uint32_t, bool in) { in ? ++nin : ++nsh; });
    int kin = lane_scan(nin, lanes, tin);
    int ksh = lane_scan(nsh, lanes, tsh);
    ksh = tin + tsh - 1 - ksh;  // the shell in reverse, as lj_list_atom leaves it
    if (t >= n) return;
    const int total = tin + tsh;
    if (total > cap) {
        if (lane == 0) {
            atomicOr(&b.bp->status, ST_NBR_OVERFLOW);
            b.nbr_cnt[base + t] = 0;
        }
        return;
    }
    walk([&](uint32_t e, bool in) { L[(size_t)(in ? kin++ : ksh--) * n] = e; });
    if (lane == 0) {
        const int padded = (total + LJ_UNROLL - 1) / LJ_UNROLL * LJ_UNROLL;
        for (int k = total; k < padded; ++k) L[(size_t)k * n] = self;
        b.nbr_cnt[base + t] = padded;
    }
}

// LANES false: an atom per thread throughout (FP32 sets that fill the GPU; with the
// other form in the kernel its registers cost 27,435 atoms 2% of a step).  FP32 with
// lanes: five blocks per SM, which leave 96 registers and no spills (2,915 atoms x 5
// images 44.9 us; 51.1 with the 72 that the compiler takes by itself.  FP64 lists, also
// of large sets, keep those: 59,999 atoms 3% of a step).
template <typename T, bool LANES>
__global__ void __launch_bounds__(TILE, LANES && sizeof(T) == 4 ? 5 : 0)
    k_lj_list(const Tile *tiles, int ntiles, BandDev *bands, int split) {
    dep_sync();
    __shared__ LJGeom<float> g;
    for (int k = blockIdx.x; k < ntiles * split; k += gridDim.x) {
        const Tile tl = tiles[k / split];
        BandDev &b = bands[tl.band];
        const ImgScalars &sc = b.sc[tl.img];
        if (b.lj_cap == 0 || !sc.rebuild) continue;  // uniform over the block
        lj_stage<float>(g, sc, *b.bp, sizeof(T) == 8, true);
        __syncthreads();
        const int lanes = sizeof(T) == 4 ? split : TILE / b.tile;  // uniform over the block
        if (!LANES || lanes == 1) {
            const int t = tile_atom(b, tl);
            if (t < b.n) lj_list_atom<T>(b, tl, g, t);
        } else if constexpr (LANES) {
            lj_list_lanes<T>(b, tl, g,
                             tl.t * b.tile + (k % split) * (TILE / split) +
                                 (int)threadIdx.x / lanes,
                             threadIdx.x % lanes, lanes);
        }
        __syncthreads();  // g is restaged for the next tile
    }
}

// List path: F_i, U_i and the virial from slot t's list entries.  The pair
// vector of an entry is (o_j - o_i) + c with c the displacement of the
// bin centres and wrap, c = C01[i0 + LJ_AXIS i1] + C2[i2] from per-axis
// tables of the image's current bin vectors built by each block in shared
// memory.  Entries are taken LJ_UNROLL at a time (lists are padded to a
// multiple of it): a group's offsets are gathered and the next group's
// entries loaded before the group's arithmetic, so a list load's latency
// overlaps a whole group of pair terms (7 blocks per SM leave the registers
// for it: measured faster than 8 without the overlap).
// MINB: resident blocks per SM the register allocation is held to (the
// autotuner picks it with the bin width: more blocks hide more gather
// latency, fewer leave more registers for the look-ahead)
template <int MINB>
__global__ void __launch_bounds__(TILE, MINB) k_lj_nbr(const Tile *tiles, BandDev *bands) {
    using T = float;
    using T4 = float4;
    const Tile tl = tiles[blockIdx.x];
    const BandDev &b = bands[tl.band];
    // no dep_sync: launched once the kernel before is complete, and letting the next
    // one in early cost it 10-18% (64 bands, 4.2e6 atom-images: 1.18 ms, 1.00 without)
    if (b.lj_cap == 0) return;  // uniform over the block: the direct path runs
    const ImgScalars &sc = b.sc[tl.img];
    __shared__ LJGeom<T> g;
    __shared__ T4 s_c01[LJ_AXIS * LJ_AXIS];
    __shared__ T4 s_c2[32];
    lj_stage(g, sc, *b.bp, false, true);
    __syncthreads();
    {
        const int L0 = 2 * (2 * g.m[0] + 1), L1 = 2 * (2 * g.m[1] + 1), L2 = 2 * (2 * g.m[2] + 1);
        for (int k = threadIdx.x; k < L0 * L1; k += TILE) {
            const int i0 = k % L0, i1 = k / L0;
            const int d0 = i0 / 2 - g.m[0], d1 = i1 / 2 - g.m[1];
            const int t0 = floor_div(d0, g.nb[0]) + (i0 & 1);
            const int t1 = floor_div(d1, g.nb[1]) + (i1 & 1);
            T4 c;
            c.x = (d0 * g.bv[0] + d1 * g.bv[3]) + (t0 * g.dh[0] + t1 * g.dh[3]);
            c.y = (d0 * g.bv[1] + d1 * g.bv[4]) + (t0 * g.dh[1] + t1 * g.dh[4]);
            c.z = (d0 * g.bv[2] + d1 * g.bv[5]) + (t0 * g.dh[2] + t1 * g.dh[5]);
            c.w = (T)0;
            s_c01[i0 + LJ_AXIS * i1] = c;
        }
        for (int k = threadIdx.x; k < L2; k += TILE) {
            const int d2 = k / 2 - g.m[2];
            const int t2 = floor_div(d2, g.nb[2]) + (k & 1);
            T4 c;
            c.x = d2 * g.bv[6] + t2 * g.dh[6];
            c.y = d2 * g.bv[7] + t2 * g.dh[7];
            c.z = d2 * g.bv[8] + t2 * g.dh[8];
            c.w = (T)0;
            s_c2[k] = c;
        }
    }
    __syncthreads();
    const int n = b.n, cap = b.lj_cap;
    const int t = tile_atom(b, tl);
    const size_t base = (size_t)tl.img * n;
    const T4 *off = (const T4 *)b.slot_off + base;
    const T rc2 = g.rc2, sig2 = g.sig2, c24 = g.c24;
    LJAcc<T> A;
    if (t < n) {
        const uint32_t *L = (const uint32_t *)b.nbr_slot + (size_t)tl.img * cap * n + t;
        const int cnt = b.nbr_cnt[base + t];  // a multiple of LJ_UNROLL
        const T4 oi = off[t];
        uint32_t e[LJ_UNROLL];  // the current group's entries
#pragma unroll
        for (int u = 0; u < LJ_UNROLL; ++u) e[u] = cnt > 0 ? L[(size_t)u * n] : 0u;
        for (int k = 0; k < cnt; k += LJ_UNROLL) {
            L += (size_t)LJ_UNROLL * n;
            T4 oj[LJ_UNROLL];
#pragma unroll
            for (int u = 0; u < LJ_UNROLL; ++u) oj[u] = off[e[u] & 0x1FFFFu];
            uint32_t en[LJ_UNROLL];
            const bool more = k + LJ_UNROLL < cnt;
#pragma unroll
            for (int u = 0; u < LJ_UNROLL; ++u) en[u] = more ? L[(size_t)u * n] : 0u;
#pragma unroll
            for (int u = 0; u < LJ_UNROLL; ++u) {
                const T4 a = s_c01[(e[u] >> 17) & 1023u], c = s_c2[e[u] >> 27];
                const T ux = (oj[u].x - oi.x) + (a.x + c.x);
                const T uy = (oj[u].y - oi.y) + (a.y + c.y);
                const T uz = (oj[u].z - oi.z) + (a.z + c.z);
                const T r2 = ux * ux + uy * uy + uz * uz;
                // r2 == 0: a padding entry (the atom itself)
                if (lj_inside(r2, rc2)) A.pair(ux, uy, uz, r2, sig2, c24);
            }
#pragma unroll
            for (int u = 0; u < LJ_UNROLL; ++u) e[u] = en[u];
        }
    }
    lj_finish(A, g, b, tl, t, t < n);
}

// The FP64 list path: bound by the FP64 pipe (~64 cycles per warp instruction),
// and in bands of few atoms by the chain of one thread's entries (31 atoms, 110
// entries each: 129 us with one thread per atom, four warps busy; 11 us with 32
// lanes.  2,915 atoms x 5 images: 146 us, now 108 us of which the FP64 pipe's
// share is 65 us).  An atom's entries are dealt to its lanes (BandDev::tile), every
// entry is screened in
// FP32 on the rounded offsets first, and only entries inside the screen (78 of
// 110; the shell entries stand last in a list, so a warp skips most of them
// together) reach FP64.
struct LJDispF {  // LJDisp rounded, for the screen
    float4 c01[LJ_C01], a[2][32], c2[32];
};
__global__ void __launch_bounds__(TILE, 4) k_lj_nbr64(const Tile *tiles, BandDev *bands) {
    using T4 = typename Vec4<double>::type;
    const Tile tl = tiles[blockIdx.x];
    const BandDev b = bands[tl.band];
    dep_sync();
    if (b.lj_cap == 0) return;  // uniform over the block: the direct path runs
    const ImgScalars &sc = b.sc[tl.img];
    __shared__ LJGeom<double> g;
    __shared__ LJDisp D;
    __shared__ LJDispF Df;
    lj_stage(g, sc, *b.bp, true, false);
    __syncthreads();
    lj_disp_stage(D, g);
    __syncthreads();
    const bool table = D.l0 * D.l1 <= LJ_C01;
    for (int k = threadIdx.x; k < LJ_C01 + 96; k += TILE) {
        const double *v = k < 64 ? D.a[k >> 5][k & 31] : k < 96 ? D.c2[k & 31] : D.c01 + 3 * (k - 96);
        if (k >= 96 && (!table || k - 96 >= D.l0 * D.l1)) break;
        const float4 f = make_float4((float)v[0], (float)v[1], (float)v[2], 0.0f);
        if (k < 64) Df.a[k >> 5][k & 31] = f;
        else if (k < 96) Df.c2[k & 31] = f;
        else Df.c01[k - 96] = f;
    }
    __syncthreads();
    const int n = b.n, cap = b.lj_cap, lanes = TILE / b.tile, lane = threadIdx.x % lanes;
    const int t = tl.t * b.tile + (int)threadIdx.x / lanes;
    const size_t base = (size_t)tl.img * n;
    const T4 *off = (const T4 *)b.slot_off + base;
    const float4 *offf = b.slot_off_lo + base;
    const double rc2 = g.rc2, sig2 = g.sig2, c24 = g.c24;
    const float screen = g.screen;
    const int l0 = D.l0;
    LJAcc<double> A;
    if (t < n) {
        const uint32_t *L = (const uint32_t *)b.nbr_slot + (size_t)tl.img * cap * n + t;
        const int cnt = b.nbr_cnt[base + t];
        const T4 oi = off[t];
        const float4 of = offf[t];
        uint32_t e = lane < cnt ? L[(size_t)lane * n] : 0u;
        for (int k = lane; k < cnt; k += lanes) {
            const uint32_t c = e;
            if (k + lanes < cnt) e = L[(size_t)(k + lanes) * n];
            const int q = (int)(c & 0x1FFFFu), i01 = (int)((c >> 17) & 1023u), i2 = (int)(c >> 27);
            const int i1 = i01 / LJ_AXIS, i0 = i01 - LJ_AXIS * i1;
            const float4 oq = offf[q], f2 = Df.c2[i2];
            float4 f;
            if (table) {
                f = Df.c01[i0 + l0 * i1];
            } else {
                const float4 fa = Df.a[0][i0], fb = Df.a[1][i1];
                f = make_float4(fa.x + fb.x, fa.y + fb.y, fa.z + fb.z, 0.0f);
            }
            const float ux = (oq.x - of.x) + (f.x + f2.x), uy = (oq.y - of.y) + (f.y + f2.y),
                        uz = (oq.z - of.z) + (f.z + f2.z);
            if (!(ux * ux + uy * uy + uz * uz < screen)) continue;
            const T4 oj = off[q];
            double x = oj.x - oi.x, y = oj.y - oi.y, z = oj.z - oi.z;
            lj_disp(D, (uint32_t)(i0 | (i1 << 5) | (i2 << 10)), x, y, z);
            const double r2 = x * x + y * y + z * z;
            // r2 == 0: a padding entry (the atom itself)
            if (lj_inside(r2, rc2)) A.pair(x, y, z, r2, sig2, c24);
        }
    }
    A.fx = lane_group_sum(A.fx, lanes);
    A.fy = lane_group_sum(A.fy, lanes);
    A.fz = lane_group_sum(A.fz, lanes);
    lj_finish(A, g, b, tl, t, t < n && lane == 0);
}

template <typename T>
void launch_lj(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s) {
    if (ntiles <= 0) return;
    launch_even(k_lj<T>, ntiles, TILE, s, tiles, bands);
}
template <typename T>
void launch_lj_list(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s) {
    if (ntiles <= 0) return;
    // a block per tile: a build walks ~370 candidates per atom, and in a
    // batch of many bands a large share of the images rebuilds at a time
    // (a capped grid was measured slower here)
    // FP32 tiles (an atom per thread) of a small set are split over several blocks
    // with as many lanes per atom: the two end images of a band, 8 to 116 tiles,
    // 125-175 us with one thread per atom
    int split = 1;
    if (sizeof(T) == 4)
        while (split < 16 && 2 * split * ntiles <= 4 * sm_count()) split *= 2;
    const int grid = ntiles * split;
    if (sizeof(T) == 4 && split == 1)
        launch_dep(k_lj_list<T, false>, grid, TILE, s, tiles, ntiles, bands, 1);
    else
        launch_dep(k_lj_list<T, true>, grid, TILE, s, tiles, ntiles, bands, split);
}
template <typename T>
void launch_lj_nbr(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s, int minb) {
    if (ntiles <= 0) return;
    if (sizeof(T) == 8) {
        launch_even(k_lj_nbr64, ntiles, TILE, s, tiles, bands);
        return;
    }
    switch (minb) {
        case 5: launch_even(k_lj_nbr<5>, ntiles, TILE, s, tiles, bands); break;
        case 6: launch_even(k_lj_nbr<6>, ntiles, TILE, s, tiles, bands); break;
        case 8: launch_even(k_lj_nbr<8>, ntiles, TILE, s, tiles, bands); break;
        default: launch_even(k_lj_nbr<7>, ntiles, TILE, s, tiles, bands); break;
    }
}
template <typename T>
void launch_energy64_lj(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s) {
    if (ntiles <= 0) return;
    k_lj_energy64<T><<<ntiles, TILE, 0, s>>>(tiles, bands);
}
template void launch_energy64_lj<float>(const Tile *, int, BandDev *, cudaStream_t);
template void launch_energy64_lj<double>(const Tile *, int, BandDev *, cudaStream_t);
template void launch_lj<float>(const Tile *, int, BandDev *, cudaStream_t);
template void launch_lj<double>(const Tile *, int, BandDev *, cudaStream_t);
template void launch_lj_list<float>(const Tile *, int, BandDev *, cudaStream_t);
template void launch_lj_list<double>(const Tile *, int, BandDev *, cudaStream_t);
template void launch_lj_nbr<float>(const Tile *, int, BandDev *, cudaStream_t, int);
template void launch_lj_nbr<double>(const Tile *, int, BandDev *, cudaStream_t, int);

}  // namespace cfneb
