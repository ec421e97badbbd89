// Shared device-side data layout of the CFNEB library.
//
// A band of N images of n atoms lives in HBM as image-major arrays:
//   X, F, Fneb, v : [ncap][n+3][3] of T   (T = double for CFNEB_FP64,
//                                           float for CFNEB_MIXED)
// rows 0..n-1 are atoms (R~ and the forces conjugate to it), rows n..n+2 the
// lattice coordinate c B (Sec. II.C: the (n+3) "atoms" of the cell filter).
// Per-image FP64 scalars (energy, virial, D, h, bin geometry) sit in
// ImgScalars[ncap]; per-band constants and FIRE state in BandParams.
//
// Kernels are launched over tile tables: each tile is (band, image, t) and
// covers atoms [t*tile, (t+1)*tile) (atom tiles: one thread per atom, tile =
// TILE, or several lanes per atom in the force kernels of small bands) or
// rows [t*rtile, (t+1)*rtile) (row tiles of the band-vector kernels, 4 or 1
// rows per thread) of that image, so any mix of bands of different sizes
// runs in one launch.  Partial sums of a tile land in a
// fixed slot (image, t) of its band, and every reduction sums the slots of a
// band in slot order: results do not depend on which other bands share the
// launch.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <stdint.h>

namespace cfneb {

constexpr int TILE = 128;           // atoms per atom tile = threads per block
constexpr int RTHREADS = 256;       // threads per block of the row-tile kernels
// Consecutive rows per thread of the row-tile kernels.  FP32: 4 (12 values, moved
// with 16-byte accesses).  FP64: 1 -- a row costs ~36 FP64 instructions in the
// dot pass, one per ~64 cycles and warp, and four of them in turn made that
// chain the pass (31 rows: band_dots 13 us, fire_update 12 us).
constexpr int rows_per_thread(size_t ts) { return ts == 4 ? 4 : 1; }
// rows per row tile (band vector kernels)
constexpr int row_tile(size_t ts) { return RTHREADS * rows_per_thread(ts); }
constexpr int MAXN_TERSOFF = 16;    // Tersoff list capacity per atom (entries within rl)
constexpr int NPART = 12;           // doubles per tile partial record
constexpr int MAX_STENCIL = 7;      // |delta| <= 7 bins per axis
// NEP-style potential: Chebyshev basis size, radial and angular functions,
// largest Legendre order, hidden units; descriptor and weight counts
constexpr int NEP_K = 6, NEP_NR = 4, NEP_NA = 2, NEP_L = 4, NEP_H = 16;
constexpr int NEP_ND = NEP_NR + NEP_NA * NEP_L;
constexpr int NEP_NW = NEP_NR * NEP_K + NEP_NA * NEP_K + NEP_H * NEP_ND + 2 * NEP_H + 1;
// offsets of cR, cA, W0, b0, w1, b1 in the flat weight array
constexpr int NEP_OCR = 0, NEP_OCA = NEP_NR * NEP_K, NEP_OW0 = NEP_OCA + NEP_NA * NEP_K,
              NEP_OB0 = NEP_OW0 + NEP_H * NEP_ND, NEP_OW1 = NEP_OB0 + NEP_H,
              NEP_OB1 = NEP_OW1 + NEP_H;
constexpr int LJ_LIST_MAX_ATOMS = 1 << 17;  // LJ list entries index 17-bit slots
// SMs of the current device (cached per device)
inline int sm_count() {
    static int cached[64] = {0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 152;
    if (!cached[dev]) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            sms <= 0)
            sms = 152;
        cached[dev] = sms;
    }
    return cached[dev];
}
// Grid of the kernels that only do work for images rebuilding their lists:
// a fixed grid (8 blocks per SM of the current device) strides over the
// tiles, so a step in which most images keep their lists costs a few reads
// per block instead of a block per tile.
inline int gated_grid() { return sm_count() * 8; }

// Launch whose blocks may become resident while the kernel before it in the
// stream drains (programmatic dependent launch, in graphs as in streams); the
// kernel calls dep_sync.  A step is a chain of ~8 kernels of 3-20 us each, the
// gaps between them a fifth of a small band's step: 384 carbon atoms 66.3 -> 58.7
// us per step, 98,303 atoms 186 -> 180 us.
template <typename... P, typename... A>
inline void launch_dep(void (*k)(P...), dim3 grid, int block, cudaStream_t s, A... a) {
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(block);
    c.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, k, static_cast<P>(a)...);
}
// The force kernels go out only once the kernel before is complete: placed among
// its last blocks, two of theirs would share an SM's arithmetic while other SMs
// idle (576 carbon atoms, FP64, 126 blocks of site terms: 85 -> 102 us per step).
template <typename... P, typename... A>
inline void launch_even(void (*k)(P...), dim3 grid, int block, cudaStream_t s, A... a) {
    k<<<grid, block, 0, s>>>(static_cast<P>(a)...);
}
// In every kernel that launch_dep starts, before its first access to anything a
// kernel writes: wait until the kernels before are complete and their writes
// visible, then let the next kernel's blocks be placed as this grid drains.  (The
// other order, placing them while this grid still waits, takes slots from it:
// 1-4 us per step slower.)  The launch tables (tiles, image references, BandDev
// records), which no kernel of a step writes, are read ahead of it: the two round
// trips to the pointers run while the kernel before drains (4 us per step).
__device__ __forceinline__ void dep_sync() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Barrier of a thread block cluster; what its threads wrote before, to shared or
// global memory, is visible to all of them after.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// potential kinds of BandParams::kind (the values of include/cfneb.h)
constexpr int KIND_LJ = 0, KIND_TERSOFF = 1, KIND_NEP = 2;

// device status bits (BandParams::status)
enum : int {
    ST_NOT_SPD = 1,
    ST_NBR_OVERFLOW = 2,
    ST_NONFINITE = 4,
};

struct ImgScalars {
    double E;            // energy (U + P Omega) of the last step's evaluation
    double U;            // potential energy
    double E64;          // FP64 energy (U + P Omega) for reporting
    double V[9];         // virial, V_eff = V - P Omega I
    double D[9];         // deformation gradient (symmetric root of B)
    double Dinv[9];
    double h[9];         // current cell h = h0 D (rows = lattice vectors)
    double hinv[9];
    double bv[9];        // bin edge vectors, row a = h_a / nb_a rounded to T
    double dh[9];        // wrap correction, row a = h_a - nb_a bv_a
    double omega;        // |det h|
    double dots[10];     // |dX+|^2, |dX-|^2, dX+.dX-, F.dX+, F.dX-, F.F, F.v,
                         // v.v, dX+.v, dX-.v (band pass 1)
    double coef[2];      // f_NEB = F + coef[0] dX+ + coef[1] dX-
    double fire[3];      // this image's F_NEB.v, |F_NEB|^2, |v|^2
    double pairs;        // neighbour entries inside the cutoff (last evaluation)
    double triples;      // ordered neighbour pairs (j, k != j) of the atoms (Tersoff)
    double Db[9];        // D when the cell list was last built (skin test)
    double dmax;         // largest |R~ - R~ at the build| of this evaluation
    long long builds;    // cell-list builds of this image slot
    long long evals;     // evaluations of this image slot
    float dfl[45];       // FP32: D hi, D lo, h hi, h lo (pairs), h0^-1 (cell list)
    float bvf[9];        // bv in FP32 (exact: bv has at most 20 significant bits)
    float dhf[9];        // dh in FP32 (the offset refresh's wrap term)
    float Dbif[9];       // FP32 inverse of Db (list reuse)
    float skin_e, skin_nD;  // the cell's part of the reuse bound (skin_terms)
    float grid, igrid;   // FP32 many-body bands: position grid and its inverse (powers of two)
    int nb[3];           // bins per axis
    int m[3];            // stencil half width per axis
    int nbins;
    int rebuild;         // this evaluation rebuilds the cell list
    unsigned int done;   // row tiles of this image finished in band pass 1
    int cell_fresh;      // D, h, Omega and the bin vectors follow the current
                         // lattice rows (set by the map-back and by the move)
};

struct TersoffParams {
    double A, B, lambda1, lambda2, beta, n, c, d, h, R, D;
};

// hi + lo = a exp(-l R), relative error below 2^-80 (host only; hi is the rounded
// value, lo = 0 where it or the exponential leaves the normal range).  Taylor's
// series to t^12 of t = -l R / 2^k, |t| < 2^-5, then k squarings, all in two-term
// sums: 5 us less per call than the host's long double exponential, which Arm
// machines do in software (three 8-atom structures in FP64, 262 -> 256 us).
struct TwoSum {
    double h, l;
};
__host__ inline TwoSum two_mul(TwoSum a, TwoSum b) {
    // (an FMA, also the first: a plain product could be fused with the sum below)
    const double p = std::fma(a.h, b.h, 0.0);
    const double e = std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h);
    const double s = p + e;
    return {s, (p - s) + e};
}
__host__ inline TwoSum scaled_exp(double a, double l, double R) {
    TwoSum t = two_mul({-l, 0.0}, {R, 0.0});
    const double plain = a * std::exp(-l * R);
    if (!(std::fabs(t.h) < 600.0)) return {plain, 0.0};
    int k = 0;
    for (; std::fabs(t.h) >= 0x1p-5; ++k) t = {0.5 * t.h, 0.5 * t.l};
    double c = 1.0;  // 12! / j!
    TwoSum r = {c, 0.0};
    for (int j = 12; j > 0; --j) {
        c *= j;
        r = two_mul(r, t);
        const double s = c + r.h;
        r = {s, ((c - s) + r.h) + r.l};
    }
    const double q = r.h / c;
    r = {q, (std::fma(-q, c, r.h) + r.l) / c};
    for (; k > 0; --k) r = two_mul(r, r);
    r = two_mul({a, 0.0}, r);
    const bool normal = std::fabs(r.h) > 0x1p-900 && std::fabs(r.h) < 0x1p1000;
    return normal ? r : TwoSum{plain, 0.0};
}

template <typename T>
struct __align__(8) TP {  // Tersoff constants in T (derived once per band, on the host)
    T A, B, l1, l2, beta, n, c2, d2, h, R, D, Rhi, pi_2D, pi_4D, inv2n, c2d2;
    T AeR, BeR;        // A exp(-l1 R), B exp(-l2 R)
    T AeRl, BeRl;      // FP64: what rounding left off (the same for every bond: in a
                       // total it does not average out)
    T R2hi, R2lo;      // R^2 as a two-term sum
    T Dlo;             // D - (T)D
    T xs;              // FP64: (beta zeta)^n below which the bond order is a series
                       // (and a whole number of 8-byte words: staged by word copies)
    // host only (std::exp of the host library): the device reads the result
    __host__ void load(const TersoffParams &p) {
        A = (T)p.A; B = (T)p.B; l1 = (T)p.lambda1; l2 = (T)p.lambda2; beta = (T)p.beta;
        n = (T)p.n; c2 = (T)(p.c * p.c); d2 = (T)(p.d * p.d); h = (T)p.h; R = (T)p.R;
        D = (T)p.D; Rhi = (T)(p.R + p.D);
        pi_2D = (T)(0.5 * 3.14159265358979323846 / p.D);
        pi_4D = (T)(0.25 * 3.14159265358979323846 / p.D);
        inv2n = (T)(0.5 / p.n);
        c2d2 = (T)(p.c * p.c / (p.d * p.d));
        AeR = (T)(p.A * std::exp(-p.lambda1 * p.R));
        BeR = (T)(p.B * std::exp(-p.lambda2 * p.R));
        AeRl = BeRl = (T)0;
        if (sizeof(T) == 8) {
            const TwoSum a = scaled_exp(p.A, p.lambda1, p.R),
                         b = scaled_exp(p.B, p.lambda2, p.R);
            AeR = (T)a.h;
            AeRl = (T)a.l;
            BeR = (T)b.h;
            BeRl = (T)b.l;
        }
        R2hi = (T)(p.R * p.R);
        R2lo = (T)(p.R * p.R - (double)R2hi);
        Dlo = (T)(p.D - (double)D);
        xs = (T)std::fmin(1.0 / 1024.0, std::fabs(p.n) / 256.0);  // x / 2n below 2^-9
    }
};


struct BandParams {
    // constants of the band
    double h0[9], h0inv[9];
    double c;            // cell factor: X_lat = c B
    double pressure;
    double k;            // spring constant
    double dt0, dt_max, maxstep;
    double rc;           // potential cutoff
    double skin;         // neighbour-list skin (0: rebuild every evaluation)
    double rl;           // list cutoff rc + skin (0 in records made before skins: rc)
    double bin_w;        // target bin width
    double ftol;         // convergence tolerance (< 0: never converged)
    double pot[12];      // LJ: LJParams; Tersoff: A, B,
                         // lambda1, lambda2, beta, n, c, d, h, R, D
    int filter, variant, climb, n;
    int N;               // current image count
    int kind;
    // FIRE state
    double dt, alpha;
    int npos, fresh;
    // outputs of the last step
    double P, FF, VV, fmax;
    double cv, cf;       // velocity mixing of the step
    long long steps;     // FIRE moves taken
    long long move_limit;// no move once steps reaches this
    int ci;              // climbing image (-1: none)
    int converged;       // fmax < ftol at the last evaluation
    int move;            // the last step moved the images
    int status;
    int stale;           // every image rebuilds at the next evaluation
    int tune_rebuild;    // rebuild at every evaluation (autotuning)
    int row_refine;      // bins along the innermost axis per bin width (>= 1)
    int pad_rr;
    // completion counter of band pass 2 (zero between launches; the last
    // block of the band resets it) and the running fmax^2 as the bits of a
    // non-negative double (ordered like the values)
    unsigned int done_b, pad_done;
    unsigned long long fmax2_bits;
    // image-range shard of a band spread over several devices: the end
    // images are neighbours' images (ghosts), the climbing image comes from
    // the caller (ci_ext: local index, or -1 for none in this range) and
    // the FIRE sums of pass 2 are left in P, FF, VV, fmax (squared) for the
    // caller to combine; the FIRE decision then takes the global sums
    int shard, ci_ext;
    TP<float> tpf;       // Tersoff constants in FP32 / FP64 (Tersoff bands)
    TP<double> tpd;
};

template <typename T> __host__ __device__ inline const TP<T> &tp_of(const BandParams &p);
template <> __host__ __device__ inline const TP<float> &tp_of<float>(const BandParams &p) {
    return p.tpf;
}
template <> __host__ __device__ inline const TP<double> &tp_of<double>(const BandParams &p) {
    return p.tpd;
}

// A bin's three indices in one int, 10 bits each (bin_grid keeps nb_a <=
// 1024): the kernels that walk a slot's stencil unpack them with shifts
// instead of dividing the linear index by the grid's extents.
__host__ __device__ inline int pack_bin(int b0, int b1, int b2) {
    return b0 | (b1 << 10) | (b2 << 20);
}
__host__ __device__ inline void unpack_bin(int p, int &b0, int &b1, int &b2) {
    b0 = p & 1023;
    b1 = (p >> 10) & 1023;
    b2 = p >> 20;
}

struct BandDev {
    int n, rows, ncap, nbins_cap;
    int atpi, rtpi;      // atom tiles / row tiles per image
    int tile;            // atoms per atom tile (TILE / lanes per atom)
    void *X, *F, *Fneb, *v;
    ImgScalars *sc;
    BandParams *bp;
    // cell list (image-major)
    int *bin_count;      // [ncap][nbins_cap]
    int *bin_start;      // [ncap][nbins_cap + 1]
    int *bin_tsum;       // [ncap][tsum_cap] scan tile sums / prefixes
    int tsum_cap;
    int *atom_bin, *atom_rank, *slot_unsorted, *slot_atom, *slot_bin, *atom_slot;  // [ncap][n]
    // (atom_bin: linear bin index; slot_bin: the bin's three indices packed
    // by pack_bin)
    void *atom_off, *slot_off;   // [ncap][n] x 4 T (x, y, z, pad): offsets, leading part
    // Offsets are FP64 or (FP32 LJ bands) FP32 from the atom's bin centre; FP32
    // many-body bands hold positions in the cell instead, as integers of the
    // image's grid (int4) and FP32 remainders (float4): see grid_split; by slot one
    // record of the two, so that a neighbour costs one 32-byte load.
    // [ncap][n] x float4.  FP32 bands: offset - leading part.  FP64 bands: the
    // offset rounded to FP32 (and the bin index), for distance screens
    float4 *atom_off_lo, *slot_off_lo;
    // neighbour-list reuse: positions and periodic wraps at the last build
    void *ref_X;         // [ncap][rows][3] T: R~ at the build (the layout of X)
    int *atom_wrap;      // [ncap][n][3]: floor(s) at the build
    int *slot_wrap;      // [ncap][n]: the wrap's place in the table of lattice shifts
    float *skin_part;    // [ncap][rtpi]: per-row-tile max displacement
    // per-slot neighbour lists: Tersoff (slot, code) pairs of MAXN_TERSOFF
    // entries, or LJ packed entries of lj_cap (0: the LJ kernel walks the
    // cell list directly)
    int lj_cap;
    int *nbr_cnt;        // [ncap][n]; many-body: | NBR_SHIFTED if a code is not CODE_ZERO
    // many-body lists: [ncap][MAXN / 4][n][4] (ent: four entries of an atom are one
    // vector); LJ lists: nbr_slot [ncap][lj_cap][n]
    int *nbr_slot;
    int *nbr_code;
    unsigned char *nbr_rev;  // entry of j's list pointing back (255: none)
    const double *nep_w;     // NEP weights [NEP_NW] in FP64 and FP32 (NEP bands)
    const float *nep_wf;
    // [ncap][MAXN][n] x 4 T: partials (x, y, z, pad).  FP64: P_ij at atom i's entry
    // j.  FP32: P_ij at the entry of atom j that points back to i, and the sum over
    // an atom's own entries in site_P [ncap][n]
    void *nbr_P;
    float4 *site_P;
    // partial sums
    int *shift;          // [ncap][27][6]: lattice shifts on the grid (FP32 many-body bands)
    double *atom_part;   // [ncap][atpi][NPART]
    double *row_part;    // [ncap][rtpi][NPART]
    // double scratch [ncap][n + 3][3]: Cartesian positions (get_path), state
    // exchange, set-up inputs
    double *cart;
};

struct Tile {
    int band, img, t, pad;
};

struct ImgRef {
    int band, img;
};

// The atom (slot) of this thread in a thread-per-atom kernel; n (none) for
// the threads past the tile's atoms.
__device__ inline int tile_atom(const BandDev &b, const Tile &tl) {
    return (int)threadIdx.x < b.tile ? tl.t * b.tile + (int)threadIdx.x : b.n;
}

// As tile_atom; in grids of more blocks than fit at a time, with the atoms of TILE /
// tile consecutive tiles on the first one's block, one per thread, and none on the
// other tiles' blocks.
__device__ inline int block_atom(const BandDev &b, const Tile &tl) {
    const int first = tl.t * b.tile;  // (tile divides TILE)
    if (gridDim.x <= 152 * 16) return tile_atom(b, tl);
    return first % TILE == 0 ? first + (int)threadIdx.x : b.n;
}

// Exclusive sum over the `lanes` consecutive lanes of a warp that share an atom
// (a power of two), and the total.  Called by whole warps.
__device__ inline int lane_scan(int v, int lanes, int &total) {
    const int l = threadIdx.x & (lanes - 1);
    int x = v;
    for (int o = 1; o < lanes; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o, lanes);
        if (l >= o) x += y;
    }
    total = __shfl_sync(0xffffffffu, x, lanes - 1, lanes);
    return x - v;
}

// Lanes that share one atom in the LJ force kernels of a band.  The band's own
// sizes decide (not its company in a batch: the order of its sums must not
// depend on it).
//
// FP64: an SM's FP64 pipe takes a warp instruction every ~16 cycles, whichever
// of its warps it comes from.  A block of TILE threads costs its share of the
// atoms' pair terms, `instr` FP64 instructions per atom, plus ~80 per thread
// for staging and reductions, and the chip takes as long as its fullest SM,
// whose k blocks keep the pipe k / (k + 0.8) busy (measured at 2 and 4).  Few
// lanes leave SMs idle, unevenly loaded or short of warps, many pay the
// overhead (lists of 14,575 atoms: 2 lanes 128 us, 4 lanes 117 us, 8 lanes
// 108 us).  152: GB300's SMs, also where fewer are visible.
inline int fp64_lanes(long long n, long long images, double instr, int least = 1) {
    int best = least;
    double cost = 1e300;
    for (int l = least; l <= 32; l *= 2) {
        const long long tile = TILE / l, blocks = (n + tile - 1) / tile * images;
        const double c = ((double)((blocks + 151) / 152) + 0.8) * (instr / l + 80.0);
        if (c < cost) {
            cost = c;
            best = l;
        }
    }
    return best;
}
inline int lanes_per_atom(long long atoms, long long want) {
    int l = 1;
    while (l < 32 && atoms * l < want) l *= 2;
    return l;
}
// FP64 instructions of an atom's LJ pair terms at the cell's mean density
inline double lj_fp64_instr(double n, double volume, double rc) {
    return 36.0 * n / volume * 4.18879020478639 * rc * rc * rc;
}
// FP32, cell walk: latency of the chained bin and offset loads; eight warps
// per scheduler hide it
constexpr long long LJ_LANES_FP32 = 152 * 4 * 32 * 8;

struct LJParams {
    double eps, sigma, rc, ephi_c;   // ephi_c = phi(rc) if shifted, else 0
    // derived on the host (an FP64 divide per block is a chain of ~20 FP64
    // instructions on one thread): sigma^2, 24 eps / sigma^2, 4 eps, rc^2
    double sig2, c24, e4, rc2;
    __host__ void derive() {
        sig2 = sigma * sigma;
        c24 = 24.0 * eps / (sigma * sigma);
        e4 = 4.0 * eps;
        rc2 = rc * rc;
    }
};


// ---- small helpers ------------------------------------------------------

__host__ __device__ inline double det3(const double *m) {
    return m[0] * (m[4] * m[8] - m[5] * m[7]) - m[1] * (m[3] * m[8] - m[5] * m[6]) +
           m[2] * (m[3] * m[7] - m[4] * m[6]);
}

__host__ __device__ inline void inv3(const double *m, double *o) {
    double d = det3(m);
    double id = 1.0 / d;
    o[0] = (m[4] * m[8] - m[5] * m[7]) * id;
    o[1] = (m[2] * m[7] - m[1] * m[8]) * id;
    o[2] = (m[1] * m[5] - m[2] * m[4]) * id;
    o[3] = (m[5] * m[6] - m[3] * m[8]) * id;
    o[4] = (m[0] * m[8] - m[2] * m[6]) * id;
    o[5] = (m[2] * m[3] - m[0] * m[5]) * id;
    o[6] = (m[3] * m[7] - m[4] * m[6]) * id;
    o[7] = (m[1] * m[6] - m[0] * m[7]) * id;
    o[8] = (m[0] * m[4] - m[1] * m[3]) * id;
}

// FP64 reciprocal and reciprocal square root from an FP32 seed and two
// Newton-Raphson steps (relative error ~1e-7 -> ~1e-14 -> ~1 ulp).  FP64
// divide and square root are long instruction sequences on this GPU; these
// serve the per-image 3x3 chains (map-back, list decisions), which run on
// one thread per image.  Arguments must lie within FP32's normal range.
__device__ inline double rcp64(double x) {
    double r = (double)(1.0f / (float)x);
    r = r * (2.0 - x * r);
    r = r * (2.0 - x * r);
    return r;
}
// Conversions made of integer operations (a conversion to or from FP64 holds
// the FP64 pipe like any FP64 instruction; integer operations issue at full
// rate), for normal values of FP32's range.
__device__ inline double f2d(float f) {  // (double)f for normal f or +-0
    const unsigned b = __float_as_uint(f), m = b & 0x7fffffffu;
    const unsigned hi = m ? (m >> 3) + 0x38000000u : 0u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(m << 29));
}
__device__ inline float d2f_pos(double x) {  // a positive x truncated to FP32
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    return __uint_as_float(((hi - 0x38000000u) << 3) | (lo >> 29));
}
// 2^-126 <= x < 2^126: x and 1 / x are normal in FP32, and __fdividef divides by x
// (by 2^126 and more it gives 0)
__device__ inline bool in_f32_range(double x) {
    return (unsigned)__double2hiint(x) - 0x38100000u < 0x47D00000u - 0x38100000u;
}
// Reciprocal of a positive x from an FP32 seed (error e ~ 2^-22) and one
// third-order step r (1 + e + e^2): ~1 ulp in three FP64 instructions; outside
// in_f32_range a divide.
__device__ inline double rcp64_pos(double x) {
    if (!in_f32_range(x)) return 1.0 / x;
    const double r = f2d(__fdividef(1.0f, d2f_pos(x)));
    const double e = fma(-x, r, 1.0);
    return fma(r, fma(e, e, e), r);
}
// sqrt(x) and 1 / sqrt(x) of a positive x: an FP32 seed and two coupled
// Newton steps (~1 ulp, nine FP64 instructions)
__device__ inline void sqrt_rcp64(double x, double &g, double &ig) {
    if (!in_f32_range(x)) {
        g = sqrt(x);
        ig = 1.0 / g;
        return;
    }
    const double y = f2d(rsqrtf(d2f_pos(x)));
    double h = 0.5 * y;
    g = x * y;
    double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    ig = 2.0 * fma(h, r, h);
}
// sin a on [0, pi/2] in FP64 by its Taylor series to the a^25 term in
// nested form (truncation below 2e-23 at pi/2); the coefficients
// 1 / ((2k)(2k + 1)) are compile-time constants (an FP64 divide is a long
// dependent sequence on this GPU)
__device__ inline double sin_quarter64(double a) {
    const double a2 = a * a;
    double p = 1.0;
#pragma unroll
    for (int k = 12; k >= 1; --k) p = 1.0 - a2 * (1.0 / (double)((2 * k) * (2 * k + 1))) * p;
    return a * p;
}
// a < b for non-negative a, b, by their bits
__device__ inline bool less_pos(double a, double b) {
    return (unsigned long long)__double_as_longlong(a) < (unsigned long long)__double_as_longlong(b);
}
__device__ inline double rsqrt64(double x) {
    double y = (double)rsqrtf((float)x);
    y = y * (1.5 - 0.5 * x * y * y);
    y = y * (1.5 - 0.5 * x * y * y);
    return y;
}
__device__ inline double sqrt64(double x) { return x > 0.0 ? x * rsqrt64(x) : 0.0; }

__host__ __device__ inline void matmul3(const double *a, const double *b, double *o) {
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            o[3 * i + j] = a[3 * i] * b[j] + a[3 * i + 1] * b[3 + j] + a[3 * i + 2] * b[6 + j];
}

template <typename T> struct Vec4;
template <> struct Vec4<float> { using type = float4; };
template <> struct Vec4<double> { using type = double4_32a; };

// FP32 offsets of one image for distance screens (list builds): an FP64
// instruction holds a warp's pipe for ~64 cycles here, so FP64 bands screen
// on their rounded copies and leave FP64 to the entries that remain.
template <typename T> __device__ inline const float4 *screen_off(const BandDev &b, size_t base) {
    return (sizeof(T) == 4 ? (const float4 *)b.slot_off : b.slot_off_lo) + base;
}
// Squared radius of such a screen that keeps every pair inside r.  The FP32
// pair vector of a rounded copy is off by at most 2^-24 of the values it is
// summed from (two offsets of about half a bin each, a bin displacement of up
// to max m bins, their sums; 4 x 2^-24 covers the three components), and a
// relative 5e-6 covers the rounding of the square.  FP32 bands screen the
// offsets they compute with: their margin is 1e-5 of r^2.
template <typename T>
__device__ inline float screen_r2(double r, const ImgScalars &sc) {
    if (sizeof(T) == 4) return (float)(r * r) * 1.00001f;
    float w = 0.0f;
    for (int k = 0; k < 9; ++k) w += fabsf(sc.bvf[k]);
    const int m = max(sc.m[0], max(sc.m[1], sc.m[2]));
    const float s = (float)r * 1.000005f + 2.4e-7f * (float)(m + 3) * w;
    return s * s;
}

// packed stencil offset: 5 bits per axis, biased by 16
__host__ __device__ inline int pack_code(int d0, int d1, int d2) {
    return (d0 + 16) | ((d1 + 16) << 5) | ((d2 + 16) << 10);
}
__host__ __device__ inline int neg_code(int code) {
    int d0 = (code & 31) - 16, d1 = ((code >> 5) & 31) - 16, d2 = ((code >> 10) & 31) - 16;
    return pack_code(-d0, -d1, -d2);
}

__device__ inline float to_float_ru(float x) { return x; }
__device__ inline float to_float_ru(double x) { return __double2float_ru(x); }

// deterministic warp sum (fixed butterfly)
__device__ inline double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// ---- lane-parallel 3x3 algebra (map-back, lattice force) -------------------
//
// One warp per image: lane l holds entry (i, j) = (l / 3, l % 3) of each
// 3x3 matrix (lanes 9..31 mirror lane l % 9; their results are unused).  A
// product is then 6 shuffles and a chain of 3 FP64 operations per lane
// instead of 27 dependent-heavy operations in one thread: the map-back is on
// the critical path of every step and FP64 latency (~64 cycles) dominates it.
struct Lane3 {
    int l, i, j;
    __device__ Lane3() : l((int)(threadIdx.x & 31) % 9), i(l / 3), j(l % 3) {}
    __device__ double eye() const { return i == j ? 1.0 : 0.0; }
};
__device__ inline double lget(double a, int src) { return __shfl_sync(0xffffffffu, a, src); }
// (A B)_ij = sum_k A_ik B_kj
__device__ inline double lmul(double a, double b, const Lane3 &p) {
    const double a0 = lget(a, 3 * p.i), a1 = lget(a, 3 * p.i + 1), a2 = lget(a, 3 * p.i + 2);
    const double b0 = lget(b, p.j), b1 = lget(b, 3 + p.j), b2 = lget(b, 6 + p.j);
    return fma(a2, b2, fma(a1, b1, a0 * b0));
}
__device__ inline double ltrans(double a, const Lane3 &p) { return lget(a, 3 * p.j + p.i); }
// cofactor C_ij = A_{i+1,j+1} A_{i+2,j+2} - A_{i+1,j+2} A_{i+2,j+1}
__device__ inline double lcof(double a, const Lane3 &p) {
    const int i1 = (p.i + 1) % 3, i2 = (p.i + 2) % 3, j1 = (p.j + 1) % 3, j2 = (p.j + 2) % 3;
    const double p11 = lget(a, 3 * i1 + j1), p22 = lget(a, 3 * i2 + j2);
    const double p12 = lget(a, 3 * i1 + j2), p21 = lget(a, 3 * i2 + j1);
    return fma(p11, p22, -(p12 * p21));
}
// det A = sum_j A_0j C_0j, in every lane
__device__ inline double ldet(double a, double c) {
    const double t = a * c;
    return lget(t, 0) + lget(t, 1) + lget(t, 2);
}

// The cell of an image from its lattice rows (Sec. II.C), one warp: lane l
// passes entry (l % 9) / 3, (l % 9) % 3 of X_lat (lanes 9..31 mirror, as
// for every lane-parallel 3x3 below).  B = X_lat / c and D = B^(1/2), the
// symmetric root, by the coupled Newton-Schulz iteration (Y -> B^(1/2),
// Z -> B^(-1/2), B scaled into the iteration's convergence region first),
// for the rotation-free filter; D = X_lat / c for the deformation gradient;
// D = I with the filter off.  Then h = h0 D, h^-1 = D^-1 h0^-1 and
// Omega = |det h|, written with D and D^-1 and their FP32 pairs into sc
// (lanes 0..8; Omega by lane 0).  Returns false, with D = I, when B (or the
// deformation gradient) is not positive definite.
// The band constants the cell needs, as one lane's share (entry l = lane %
// 9 of h0 and h0^-1): loaded together, ahead of the FP64 work.
struct CellIn {
    int filter, variant;
    double c, h0, h0inv;
};
__device__ inline CellIn cell_in(const BandParams *bp) {
    const int l = (int)(threadIdx.x & 31) % 9;
    return {bp->filter, bp->variant, bp->c, bp->h0[l], bp->h0inv[l]};
}

__device__ inline bool image_cell_warp(const CellIn &k, double xlat, ImgScalars &sc,
                                       double &h_out) {
    const Lane3 p;
    const int lane = threadIdx.x & 31;
    double D = p.eye(), Di = p.eye();
    bool ok = true;
    if (k.filter) {
        // lattice rows are stored as c (B - I) (or c (D - I)): B = X / c + I
        const double L = xlat * rcp64(k.c) + p.eye();
        if (k.variant == 0) {
            const double B = 0.5 * (L + ltrans(L, p));
            const double C = lcof(B, p);
            const double det = ldet(B, C);
            // Sylvester's criterion: B00 > 0, the leading 2x2 minor (= C22) > 0, det > 0
            ok = lget(B, 0) > 0.0 && lget(C, 8) > 0.0 && det > 0.0;
            if (ok) {
                // spectrum bracket [det / g^2, g], g = largest Gershgorin row bound
                const double rs = fabs(lget(B, 3 * p.i)) + fabs(lget(B, 3 * p.i + 1)) +
                                  fabs(lget(B, 3 * p.i + 2));
                const double g = fmax(fmax(lget(rs, 0), lget(rs, 3)), lget(rs, 6));
                const double ig = rcp64(g);
                const double mu = 0.5 * (g + det * ig * ig);
                double Y = B * rcp64(mu), Z = p.eye();
                for (int it = 0; it < 40; ++it) {
                    const double e = p.eye() - lmul(Z, Y, p);  // I - Z Y
                    const double Tm = p.eye() + 0.5 * e;       // (3I - Z Y) / 2
                    float dev = fabsf((float)e);
                    for (int o = 16; o > 0; o >>= 1)
                        dev = fmaxf(dev, __shfl_xor_sync(0xffffffffu, dev, o));
                    const double Y1 = lmul(Y, Tm, p), Z1 = lmul(Tm, Z, p);
                    Y = Y1;
                    Z = Z1;
                    if (dev < 1e-9f) break;  // the last step took it to ~1e-18
                }
                const double rmu = sqrt64(mu);
                D = 0.5 * (Y + ltrans(Y, p)) * rmu;
                Di = 0.5 * (Z + ltrans(Z, p)) * rcp64(rmu);
            }
        } else {
            const double C = lcof(L, p);
            const double det = ldet(L, C);
            ok = det > 0.0;
            if (ok) {
                D = L;
                Di = ltrans(C, p) * rcp64(det);
            }
        }
    }
    if (!ok) D = Di = p.eye();
    const double h = lmul(k.h0, D, p);
    const double hinv = lmul(Di, k.h0inv, p);  // (h0 D)^-1 = D^-1 h0^-1
    const double omega = fabs(ldet(h, lcof(h, p)));
    if (lane < 9) {
        sc.D[lane] = D;
        sc.Dinv[lane] = Di;
        sc.h[lane] = h;
        sc.hinv[lane] = hinv;
        // FP32 pairs of D and h and FP32 h0^-1 for the FP32 cell-list path
        const float Dh = (float)D, hh = (float)h;
        sc.dfl[lane] = Dh;
        sc.dfl[9 + lane] = (float)(D - (double)Dh);
        sc.dfl[18 + lane] = hh;
        sc.dfl[27 + lane] = (float)(h - (double)hh);
        sc.dfl[36 + lane] = (float)k.h0inv;
    }
    if (lane == 0) sc.omega = omega;
    h_out = h;
    return ok;
}

// ---- positions on an integer grid (FP32 many-body bands) --------------------
//
// The many-body forces need pair vectors to well below FP32's resolution of a
// position.  Each atom's position in the cell (R minus the lattice vectors it
// was wrapped by at the list build) is an integer triple of a power-of-two grid
// g plus an FP32 remainder of at most g / 2.  A pair's leading part is then an
// exact integer difference that converts to FP32 exactly (|r| < 2^24 g), its
// low part a difference of remainders (~2^-24 g), and a periodic image adds a
// lattice shift of the same form: no bin centres, bin displacements or wrap
// corrections, which took ~190 of a Tersoff atom's ~1,770 instructions (98,303
// atoms x 9 images: site terms 83.8 -> 79.8 us, offset refresh 21.1 -> 18.0 us;
// the table below costs the moving warp 0.6 us, which small bands see).
// g is the least power of two with 1.25 times the cell's extent below 2^30 g and rl
// below 2^24 g / 1.1: 2^-22 A for carbon's 2.25 A lists in cells up to 204 A, 2^-21 A
// up to 409 A, and so on; the remainders keep the precision.
constexpr int SHIFTS = 27;  // lattice shifts t_a in {-1, 0, 1}; others are formed on the fly
struct F2 {  // unevaluated sum hi + lo of two floats
    float hi, lo;
};
// a (hi + lo) exactly up to the rounding of the low product
__device__ inline F2 f2_mul(float a, float bh, float bl) {
    const float p = __fmul_rn(a, bh);
    float e = fmaf(a, bh, -p);
    e = fmaf(a, bl, e);
    return {p, e};
}
__device__ inline F2 f2_add(F2 a, F2 b) {
    const float s = __fadd_rn(a.hi, b.hi);
    const float bb = __fsub_rn(s, a.hi);
    float e = __fadd_rn(__fsub_rn(a.hi, __fsub_rn(s, bb)), __fsub_rn(b.hi, bb));
    e = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
    const float hi = __fadd_rn(s, e);
    return {hi, __fsub_rn(e, __fsub_rn(hi, s))};
}
// v = i g + lo, |v| < 2^33 g, i modulo 2^32.  Rounding by adding 1.5 2^23 (a
// rintf and a conversion per step would queue at 16 lanes per clock and SM): in
// units of g, v.hi gives a multiple of 4096 and an exact rest; the rest is a
// multiple of v.hi's last place and v.lo at most half of one, so their
// fast two-sum is exact.  A non-finite v ends in lo.
__device__ inline void grid_split(F2 v, float g, float ig, int &i, float &lo) {
    const float M = 12582912.0f;  // 1.5 2^23 = 0x4B400000
    const float u = v.hi * ig, w = v.lo * ig;
    const float a = __fadd_rn(u * (1.0f / 4096.0f), M);
    const float rest = fmaf(__fsub_rn(a, M), -4096.0f, u);
    const float s = __fadd_rn(rest, w), e = __fsub_rn(w, __fsub_rn(s, rest));
    const float k = __fadd_rn(s, M);
    i = (int)(((unsigned)__float_as_int(a) - 0x4B400000u) * 4096u +
              ((unsigned)__float_as_int(k) - 0x4B400000u));
    lo = __fadd_rn(__fsub_rn(s, __fsub_rn(k, M)), e) * g;
}
// exponent of a positive normal x, and 2^e
__device__ inline int expo(float x) { return (__float_as_int(x) >> 23) - 127; }
__device__ inline float pow2f(int e) { return __int_as_float((min(max(e, -126), 127) + 127) << 23); }
// The lattice shift t on the grid, from the FP32 pairs of h
__device__ inline void lattice_shift(const float *hh, const float *hl, float g, float ig, int t0,
                                     int t1, int t2, int (&s)[3], float (&lo)[3]) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        F2 v = f2_mul((float)t0, hh[c], hl[c]);
        v = f2_add(v, f2_mul((float)t1, hh[3 + c], hl[3 + c]));
        v = f2_add(v, f2_mul((float)t2, hh[6 + c], hl[6 + c]));
        grid_split(v, g, ig, s[c], lo[c]);
    }
}
// The grid of an image's cell and its table of lattice shifts (one warp; h =
// entry lane % 9 of the cell, rl = the list cutoff).  On the move's critical
// path: the cell's entries go round by shuffles, not through memory.
static __device__ __noinline__ void grid_warp(ImgScalars &sc, int *shift, double h, float rl) {
    const int lane = threadIdx.x & 31;
    const float mh = (float)h, ml = (float)(h - (double)mh);
    float hh[9], hl[9], ext = 0.0f;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
        hh[k] = __shfl_sync(0xffffffffu, mh, k);
        hl[k] = __shfl_sync(0xffffffffu, ml, k);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) ext = fmaxf(ext, fabsf(hh[c]) + fabsf(hh[3 + c]) + fabsf(hh[6 + c]));
    // 2^e > 1.25 ext (room for drift between builds)
    const int e = max(expo(1.25f * ext) + 1 - 30, expo(1.1f * rl) + 1 - 24);
    const float g = pow2f(e), ig = pow2f(-e);
    if (lane < SHIFTS) {
        int s[3];
        float lo[3];
        lattice_shift(hh, hl, g, ig, lane % 3 - 1, (lane / 3) % 3 - 1, lane / 9 - 1, s, lo);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            shift[6 * lane + c] = s[c];
            shift[6 * lane + 3 + c] = __float_as_int(lo[c]);
        }
    }
    if (lane == 0) {
        sc.grid = g;
        sc.igrid = ig;
    }
}

// Bin vectors of the image's grid for its current cell, one entry per lane
// (lanes 0..8; the whole warp calls): bv_a on a grid of q = 2^(e - 19),
// 2^e >= max |h_a / nb_a|, so every sum of three products delta_a bv_a
// (|delta| <= 7) is exact in FP32; dh = h - nb bv carries the (sub-1e-4 A)
// quantisation to the periodic wrap.  Only the binade of max |h_a / nb_a|
// matters; found in FP32 it can be one binade low by an ulp, and then
// |bv| <= (2^19 + 1) q: three terms |delta| <= 7 still sum below 2^24 q.
// nba = sc.nb[(lane % 9) / 3] and h = sc.h[lane % 9] are passed in (lanes
// 9..31 mirror lane % 9; only lanes 0..8 store).
__device__ inline void bin_vectors_warp(ImgScalars &sc, int nba, double h) {
    const int lane = threadIdx.x & 31;
    const int l = lane % 9;
    float bmax = fabsf((float)h / (float)nba);
    for (int o = 16; o > 0; o >>= 1) bmax = fmaxf(bmax, __shfl_xor_sync(0xffffffffu, bmax, o));
    const int e = ilogbf(bmax) + 1 - 19;
    const double q = ldexp(1.0, e), iq = ldexp(1.0, -e);  // exact powers of two
    const double v = q * rint(h * rcp64((double)nba) * iq);
    if (lane < 9) {
        sc.bv[l] = v;
        sc.bvf[l] = (float)v;
        sc.dh[l] = h - nba * v;
        sc.dhf[l] = (float)(h - nba * v);
    }
}

// upper bound of the spectral norm of a 3x3 matrix: the smaller of the
// Frobenius norm and sqrt(|A|_1 |A|_inf), in FP32 and raised by 1e-6 to
// stay a bound
__device__ inline float norm2_bound(const float *A) {
    float f = 0.0f, c1 = 0.0f, ci = 0.0f;
    for (int i = 0; i < 3; ++i) {
        float rs = 0.0f, cs = 0.0f;
        for (int j = 0; j < 3; ++j) {
            f += A[3 * i + j] * A[3 * i + j];
            rs += fabsf(A[3 * i + j]);
            cs += fabsf(A[3 * j + i]);
        }
        ci = fmaxf(ci, rs);
        c1 = fmaxf(c1, cs);
    }
    return fminf(sqrtf(f), sqrtf(c1 * ci)) * 1.000001f;
}

// FP32 inverse of a 3x3 matrix (cofactors over the determinant)
__device__ inline void inv3f(const float *m, float *o) {
    const float c00 = m[4] * m[8] - m[5] * m[7], c01 = m[5] * m[6] - m[3] * m[8],
                c02 = m[3] * m[7] - m[4] * m[6];
    const float id = 1.0f / (m[0] * c00 + m[1] * c01 + m[2] * c02);
    o[0] = c00 * id;
    o[1] = (m[2] * m[7] - m[1] * m[8]) * id;
    o[2] = (m[1] * m[5] - m[2] * m[4]) * id;
    o[3] = c01 * id;
    o[4] = (m[0] * m[8] - m[2] * m[6]) * id;
    o[5] = (m[2] * m[3] - m[0] * m[5]) * id;
    o[6] = c02 * id;
    o[7] = (m[1] * m[6] - m[0] * m[7]) * id;
    o[8] = (m[0] * m[4] - m[1] * m[3]) * id;
}

// The cell's part of the list-reuse bound (one thread): with M = D_b^-1 D - I
// (D_b = D at the build), skin_e = |M|_2 bound and skin_nD = |D|_2 bound, in
// FP32: M - I is small, so its FP32 rounding (~1e-7 absolute) moves the
// bound by far less than the 1e-5 margins, which also cover the FP32 list
// test and displacement.  D from its FP32 leading part, D_b^-1 from the
// build (Dbi: sc.Dbif, or a copy of it loaded ahead).
__device__ inline void skin_terms(ImgScalars &sc, const float *Dbi) {
    const float *D = sc.dfl;
    float M[9];
    for (int i = 0; i < 3; ++i)
        for (int j = 0; j < 3; ++j)
            M[3 * i + j] = Dbi[3 * i] * D[j] + Dbi[3 * i + 1] * D[3 + j] +
                           Dbi[3 * i + 2] * D[6 + j] - (i == j ? 1.0f : 0.0f);
    sc.skin_e = norm2_bound(M) * 1.00001f + 1e-6f;
    sc.skin_nD = norm2_bound(D);
}

// FP64 sums of K values over `count` records (value k of record q at
// rec[q * stride + k]) in a fixed order that needs few FP64 instructions (an
// FP64 instruction occupies a warp's FP64 pipe for ~64 cycles here, so
// butterflies over many warps cost more than the sums themselves): thread
// k + K g (g < G) adds value k of records g, g + G, g + 2G, ... in turn, and
// thread k (< K) then adds the G partial sums in order and returns total k.
// Needs blockDim.x >= K G; every thread of the block must call it.
template <int K, int G>
__device__ inline double block_sum_records(const double *rec, int stride, int count) {
    __shared__ double s_part[G * K];
    const int tid = threadIdx.x;
    if (tid < K * G) {
        // four interleaved accumulators (records g, g + G, g + 2G, g + 3G go
        // to accumulators 0..3 in turn): a quarter of the dependent FP64 add
        // chain, with the loads of each round in flight together
        const int k = tid % K, g = tid / K;
        double v0 = 0.0, v1 = 0.0, v2 = 0.0, v3 = 0.0;
        int q = g;
        for (; q + 3 * G < count; q += 4 * G) {
            v0 += rec[(size_t)q * stride + k];
            v1 += rec[(size_t)(q + G) * stride + k];
            v2 += rec[(size_t)(q + 2 * G) * stride + k];
            v3 += rec[(size_t)(q + 3 * G) * stride + k];
        }
        if (q < count) v0 += rec[(size_t)q * stride + k];
        if (q + G < count) v1 += rec[(size_t)(q + G) * stride + k];
        if (q + 2 * G < count) v2 += rec[(size_t)(q + 2 * G) * stride + k];
        s_part[g * K + k] = (v0 + v1) + (v2 + v3);
    }
    __syncthreads();
    double tot = 0.0;
    if (tid < K)
        for (int g = 0; g < G; ++g) tot += s_part[g * K + tid];
    __syncthreads();
    return tot;
}

// FP64 sums of K values over `count` records like block_sum_records, with
// the loads in flight together: thread k + K g (g < G = NT / K) loads value
// k of records g, g + G, ..., g + (U - 1) G at once and adds them in that
// order (U G records per round trip instead of a chain of four), then the
// G partial sums are added in H = 8 strided groups and the groups in
// order.  The FP64 add count is the same; the round trips fall from
// count / 4G to count / UG.  CG: loads bypass L1 (records written by other
// blocks of the running kernel).  NT = blockDim.x; every thread calls.
template <int K, int U, int NT, bool CG>
__device__ inline double block_sum_records_wide(const double *rec, int stride, int count) {
    constexpr int G = NT / K, H = 8;
    static_assert(G >= H, "too few threads for the group sums");
    __shared__ double s_part[G * K];
    __shared__ double s_grp[H * K];
    const int tid = threadIdx.x;
    if (tid < K * G) {
        const int k = tid % K, g = tid / K;
        double v = 0.0;
        for (int q0 = g; q0 < count; q0 += U * G) {
            double w[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int q = q0 + u * G;
                const double *p = rec + (size_t)q * stride + k;
                w[u] = q < count ? (CG ? __ldcg(p) : *p) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; ++u) v += w[u];
        }
        s_part[g * K + k] = v;
    }
    __syncthreads();
    if (tid < K * H) {
        const int k = tid % K, h = tid / K;
        double v = 0.0;
        for (int g = h; g < G; g += H) v += s_part[g * K + k];
        s_grp[h * K + k] = v;
    }
    __syncthreads();
    double tot = 0.0;
    if (tid < K)
        for (int h = 0; h < H; ++h) tot += s_grp[h * K + tid];
    __syncthreads();
    return tot;
}

// Sum K per-thread values over a TILE-thread block in FP64 (fixed order);
// thread 0 of the block receives the totals in out[0..K-1].
template <int K>
__device__ inline void block_sum(double (&v)[K], double *out) {
    __shared__ double red[TILE / 32][K > 0 ? K : 1];
    int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        double s = warp_sum(v[k]);
        if (lane == 0) red[w][k] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            double s = 0.0;
            for (int q = 0; q < TILE / 32; ++q) s += red[q][k];
            out[k] = s;
        }
    }
    __syncthreads();  // red[] may be reused by a later call
}

// Sum K per-thread values of type T over a TILE-thread block: within each warp in T
// (fixed butterfly), across warps in FP64.  With T = float the long accumulations
// (across warps, tiles and images) stay FP64 while the per-element work avoids FP64
// arithmetic.  The totals go to dst[0..K-1]: lane k of warp 0 sums value k across the
// warps, so the FP64 additions take K/32 warp instructions instead of K in thread 0
// (an FP64 instruction occupies a warp's FP64 pipe for ~64 cycles here).
template <int K, typename T>
__device__ inline void block_sum_store(T (&v)[K], double *dst) {
    static_assert(K <= 32, "one lane per value");
    __shared__ T red[TILE / 32][K > 0 ? K : 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        T s = v[k];
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) red[w][k] = s;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int q = 0; q < TILE / 32; ++q) s += (double)red[q][threadIdx.x];
        dst[threadIdx.x] = s;
    }
    __syncthreads();
}

// As block_sum_store for K <= 16 values, with a transposing warp reduction:
// at each butterfly level a lane keeps half of its values and adds the
// partner's copy of that half (16 shuffles in all instead of 5 per value),
// so lane l ends with the warp total of value l >> 1.  Fixed order; the
// totals go to dst[0..K-1] in FP64 (across the warps, in warp order).
template <int K, typename T>
__device__ inline void block_sum_store_tr(const T (&v)[K], double *dst) {
    static_assert(K <= 16, "values are padded to 16");
    __shared__ T red[TILE / 32][16];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    T a[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) a[k] = k < K ? v[k] : (T)0;
#pragma unroll
    for (int h = 8, o = 16; h >= 1; h >>= 1, o >>= 1) {
        const bool hi = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < h; ++k) {
            const T send = hi ? a[k] : a[k + h];
            const T keep = hi ? a[k + h] : a[k];
            a[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    a[0] += __shfl_xor_sync(0xffffffffu, a[0], 1);
    if ((lane & 1) == 0) red[w][lane >> 1] = a[0];
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0.0;
        for (int q = 0; q < TILE / 32; ++q) s += (double)red[q][threadIdx.x];
        dst[threadIdx.x] = s;
    }
    __syncthreads();
}

// Sum K per-thread values over a block of any multiple of 32 threads (up to
// 1024) in FP64, fixed order (a warp butterfly within each warp, then one
// across the warp totals); thread 0 receives the totals.  Butterflies keep
// the dependent FP64 chain at 5 + 5 additions (a dependent FP64 operation
// costs ~64 cycles here).
template <int K>
__device__ inline void block_sum_any(double (&v)[K], double *out) {
    __shared__ double red[32][K];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const double s = warp_sum(v[k]);
        if (lane == 0) red[w][k] = s;
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const double s = warp_sum(lane < nw ? red[lane][k] : 0.0);
            if (lane == 0) out[k] = s;
        }
    }
    __syncthreads();
}

// threads of the per-image / per-band reduction kernels
constexpr int RED_THREADS = 256;
// threads of the per-image finalize (one block per image: wide record sums)
constexpr int FIN_THREADS = 1024;

// Copy a record between global and shared memory with all threads of the
// block (8-byte words).  The per-image and per-band kernels read many fields
// of ImgScalars and BandParams on one thread; staged first, those reads cost
// one round trip instead of a chain of dependent global loads.
template <typename S>
__device__ inline void stage_copy(S *dst, const S *src) {
    static_assert(sizeof(S) % 8 == 0, "record size must be a multiple of 8 bytes");
    static_assert(alignof(S) >= 8, "record must be 8-byte aligned for word copies");
    // every word loaded before the first store (the compiler cannot tell
    // the shared side from the global one, so interleaved copies would wait
    // out one round trip per word); PER words per thread cover the record
    // for any block of at least 32 threads
    constexpr int NW = (int)(sizeof(S) / 8), PER = (NW + 31) / 32;
    const unsigned long long *s = (const unsigned long long *)src;
    unsigned long long *d = (unsigned long long *)dst;
    unsigned long long w[PER];
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = threadIdx.x + k * blockDim.x;
        w[k] = i < NW ? s[i] : 0ull;
    }
#pragma unroll
    for (int k = 0; k < PER; ++k) {
        const int i = threadIdx.x + k * blockDim.x;
        if (i < NW) d[i] = w[k];
    }
}

// ---- many-body lists ---------------------------------------------------------

// FP32 bands: an image's position grid and its table of lattice shifts, staged
// by the block.  An entry's code is its lattice shift (t0, t1, t2) as packed by
// pack_code; CODE_ZERO: none.
struct GridF {
    float g, ig;
    int4 s[SHIFTS];     // shift on the grid
    float4 lo[SHIFTS];  // its remainder
};
constexpr int CODE_ZERO = 16 | (16 << 5) | (16 << 10);
constexpr int NBR_SHIFTED = 256, NBR_COUNT = 255;
// Place of entry k of atom t in an image's many-body list
__device__ inline size_t ent(int k, int t, int n) { return ((size_t)(k >> 2) * n + t) * 4 + (k & 3); }
__device__ inline void grid_stage(GridF &G, const BandDev &b, int img) {
    const int *sh = b.shift + (size_t)img * SHIFTS * 6;
    if (threadIdx.x < SHIFTS) {
        const int *p = sh + 6 * threadIdx.x;
        G.s[threadIdx.x] = make_int4(p[0], p[1], p[2], 0);
        G.lo[threadIdx.x] = make_float4(__int_as_float(p[3]), __int_as_float(p[4]),
                                        __int_as_float(p[5]), 0.0f);
    }
    if (threadIdx.x == 32) G.g = b.sc[img].grid;
    if (threadIdx.x == 33) G.ig = b.sc[img].igrid;
}
// A slot's position record: integers (as float bits) and remainders
__device__ __forceinline__ void load_pos(const float4 *p, float4 &i, float4 &lo) {
    asm("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
        : "=f"(i.x), "=f"(i.y), "=f"(i.z), "=f"(i.w), "=f"(lo.x), "=f"(lo.y), "=f"(lo.z), "=f"(lo.w)
        : "l"(p)
        : "memory");
}
__device__ inline int grid_diff(float a, float b) { return __float_as_int(a) - __float_as_int(b); }

// The shift of a code: the table's, or (cells narrower than the list cutoff)
// formed from the cell
__device__ inline void grid_shift(const GridF &G, const ImgScalars &sc, int code, int (&s)[3],
                                  float (&lo)[3]) {
    const int t0 = (code & 31) - 16, t1 = ((code >> 5) & 31) - 16, t2 = ((code >> 10) & 31) - 16;
    if ((unsigned)(t0 + 1) <= 2u && (unsigned)(t1 + 1) <= 2u && (unsigned)(t2 + 1) <= 2u) {
        const int k = (t0 + 1) + 3 * (t1 + 1) + 9 * (t2 + 1);
        s[0] = G.s[k].x; s[1] = G.s[k].y; s[2] = G.s[k].z;
        lo[0] = G.lo[k].x; lo[1] = G.lo[k].y; lo[2] = G.lo[k].z;
    } else {
        lattice_shift(sc.dfl + 18, sc.dfl + 27, G.g, G.ig, t0, t1, t2, s, lo);
    }
}

// Bin offset and periodic wrap of a stencil code from bin (b0, b1, b2)
__device__ inline void ters_code(int code, int b0, int b1, int b2, const int *s_nb, int (&d)[3],
                                 int (&t)[3]) {
    const int b[3] = {b0, b1, b2};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        d[a] = ((code >> (5 * a)) & 31) - 16;
        int w = b[a] + d[a];
        t[a] = 0;
        while (w < 0) { w += s_nb[a]; --t[a]; }
        while (w >= s_nb[a]) { w -= s_nb[a]; ++t[a]; }
    }
}

// b = (1 + x)^(-1/2n) for x = (beta zeta)^n: below xs (2^-10, carbon: x ~ 1e-4; less
// where n < 1/4, so that u = x / 2n stays below 2^-9) by the series of log(1 + x) to
// x^6 and exp(-u) to u^5 (truncation below 1e-18 relative)
__device__ inline double bond_order_x(double x, double inv2n, double xs) {
    if (x < xs) {
        const double l = x * (1.0 - x * (0.5 - x * (1.0 / 3.0 - x * (0.25 - x * (0.2 - x * (1.0 / 6.0))))));
        const double u = inv2n * l;
        return 1.0 - u * (1.0 - u * (0.5 - u * (1.0 / 6.0 - u * (1.0 / 24.0 - u * (1.0 / 120.0)))));
    }
    return exp(-inv2n * log1p(x));
}

// ---- launchers (defined in the kernel translation units) ---------------

// map-back and the cell-list decision of every image (the displacements
// since the last build come from the last move, per row tile); force: every
// image, or the band's end images, whose rows a caller may have replaced,
// rebuild whatever the decision
enum : int { REBUILD_ASKED = 0, REBUILD_ALL = 1, REBUILD_ENDS = 2 };
template <typename T>
void launch_mapback(const ImgRef *imgs, int count, BandDev *bands, int force, cudaStream_t s);
// bins or offsets; with has_cond also sets `cond` (a conditional graph
// node's handle, default 0) to 1 when a listed image rebuilds its cell list
template <typename T>
void launch_bin_assign(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s,
                       cudaGraphConditionalHandle cond = 0, int has_cond = 0);
// part 0: tile sums, 1: scan of the tile sums, 2: final per-bin scan
void launch_bin_scan(const ImgRef *imgs, int count, int max_bins, BandDev *bands,
                     cudaStream_t s, int part);
void launch_bin_scatter(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
// Images that k_bin_sort takes (cell.cu)
constexpr int SORT_CL = 8, SORT_THREADS = 512, SORT_BINS = 16384;
constexpr int SORT_ATOMS = 28672, SORT_CAP = 8 * SORT_BINS;
template <typename T>
void launch_bin_sort(const ImgRef *imgs, int count, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_bin_order(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_lj(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_lj_list(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
// minb: resident blocks per SM of the force kernel variant (FP32: 5-8 for
// LJ, 4-8 for Tersoff; the autotuner picks it)
template <typename T>
void launch_lj_nbr(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s, int minb);
template <typename T>
void launch_tersoff_list(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_tersoff_reverse(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_tersoff_partials(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s,
                             int minb);
template <typename T>
void launch_nep_partials(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_tersoff_gather(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_image_finalize(const ImgRef *imgs, int count, BandDev *bands, cudaStream_t s);
// band pass 1 (dots, then per image and per band the NEB coefficients and
// FIRE sums), pass 2 (f_NEB, fmax, FIRE decision); the dots alone and their
// per-image sums (spacings of the refinement check)
template <typename T>
void launch_band_dots(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_neb_force(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_band_dots_only(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
void launch_dots_reduce(const ImgRef *imgs, int count, BandDev *bands, cudaStream_t s);
// the FIRE decision of a shard on the global sums (P, F.F, v.v, fmax^2)
void launch_shard_fire(BandDev *band, double P, double FF, double VV, double fmax2,
                       cudaStream_t s);
template <typename T>
void launch_fire_update(const Tile *tiles, int ntiles, const ImgRef *imgs, int nimg,
                        BandDev *bands, cudaStream_t s);
// FP64 energies for reporting: per-tile sums (LJ bands / many-body bands),
// then the images' totals
template <typename T>
void launch_energy64_lj(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_energy64(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
void launch_energy_finalize(const ImgRef *imgs, int nimg, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_cartesian(int N, int n, BandDev *band, cudaStream_t s);
template <typename T>
void launch_midpoint(BandDev *band, int img, int rows, cudaStream_t s);
void launch_gather_status(BandDev *bands, int nb, double *out, cudaStream_t s);
struct Mat3 {
    double m[9];
};
template <typename T>
void launch_setup(const double *R0, const double *R1, const double *noise, int n, int N,
                  BandDev *band, cudaStream_t s, const Mat3 &h1);
// Single points: image 0 of every tile's band from the Cartesian positions in
// BandDev::cart (R~ = R: the reference cell is the structure's own), and its
// forces back into them
template <typename T>
void launch_points_load(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
template <typename T>
void launch_points_store(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s);
// Vectors [N][n + 3][3] of doubles in BandDev::cart to and from the band's
// padded rows (which: 0 X, 1 F, 2 f_NEB; X with the lattice rows c B of the C
// ABI, f_NEB with zero end images)
template <typename T>
void launch_state_load(BandDev *band, int N, int n, double c, cudaStream_t s);
template <typename T>
void launch_state_store(BandDev *band, int which, int N, int n, double c, cudaStream_t s);
// FIRE restart and stale lists; tolerance and move budget
void launch_fire_reset(BandDev *band, cudaStream_t s);
void launch_set_control(BandDev *band, double ftol, long long move_limit, cudaStream_t s);

}  // namespace cfneb
