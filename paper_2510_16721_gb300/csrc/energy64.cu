// FP64 total energies for reporting (paths, barriers, single points).
//
// The per-step force kernels of the mixed path evaluate per-atom energies in
// FP32; that is enough to order neighbouring images for the upwind tangent
// and to pick the climbing image, but a total over ~1e5 atoms carries errors
// of ~1e-2 eV (in a perfect crystal every atom makes the same rounding
// error).  Reported energies therefore come from these kernels, which redo
// the energy -- and only the energy -- in FP64 from the neighbour lists of the
// configuration being reported: pair vectors in FP64 (entries64), then the Tersoff
// or NEP-style energy of Sec. II.B's per-atom split (Lennard-Jones: k_lj_energy64,
// beside its force kernels) summed over atoms in FP64.  Used by cfneb_get_path and,
// in mixed precision, by cfneb_evaluate, never inside a relaxation step.
//
// FP64 arithmetic is scarce on this GPU, so it is spent on the terms only:
// the atom's neighbour list (rebuilt with the cell list) is walked instead of
// the stencil.
#include "common.cuh"

namespace cfneb {

// Unit vectors, lengths and their inverses of the neighbour-list entries of
// slot t within rc (periodic images included, the atom itself excluded), in
// FP64; returns their count.  FP32 bands: grid differences are exact in FP32
// and converted by integer operations, the remainders join with one FP64
// addition.  FP64 bands: bin displacements exact in FP32, wraps where there are
// any.
struct Entries64 {
    double x[MAXN_TERSOFF], y[MAXN_TERSOFF], z[MAXN_TERSOFF], r[MAXN_TERSOFF];
};
__device__ inline bool add_entry(Entries64 &E, int k, double x, double y, double z, double rc2) {
    const double r2 = x * x + y * y + z * z;
    if (!(r2 < rc2 && r2 > 0.0)) return false;
    double r, ir;
    sqrt_rcp64(r2, r, ir);
    E.x[k] = x * ir;
    E.y[k] = y * ir;
    E.z[k] = z * ir;
    E.r[k] = r;
    return true;
}
__device__ inline int entries64(const BandDev &b, const Tile &tl, int t, double rc,
                                const GridF &G, Entries64 &E, float) {
    const ImgScalars &sc = b.sc[tl.img];
    const size_t base = (size_t)tl.img * b.n;
    const float4 *pos = (const float4 *)b.slot_off + 2 * base;
    const int *nslot = b.nbr_slot + base * MAXN_TERSOFF;
    const int *ncode = b.nbr_code + base * MAXN_TERSOFF;
    const int ne = b.nbr_cnt[base + t] & NBR_COUNT;
    float4 pi, li;
    load_pos(pos + 2 * t, pi, li);
    int cnt = 0;
    for (int e = 0; e < ne; ++e) {
        const int q = nslot[ent(e, t, b.n)], code = ncode[ent(e, t, b.n)];
        float4 pj, lj;
        load_pos(pos + 2 * q, pj, lj);
        int s[3] = {0, 0, 0};
        float lo[3] = {0.0f, 0.0f, 0.0f};
        if (code != CODE_ZERO) grid_shift(G, sc, code, s, lo);
        const auto component = [&](float j, float i, float jl, float il, int c) {
            return f2d((float)(grid_diff(j, i) + s[c]) * G.g) + f2d((jl - il) + lo[c]);
        };
        const double x = component(pj.x, pi.x, lj.x, li.x, 0);
        const double y = component(pj.y, pi.y, lj.y, li.y, 1);
        const double z = component(pj.z, pi.z, lj.z, li.z, 2);
        cnt += add_entry(E, cnt, x, y, z, rc * rc);
    }
    return cnt;
}
__device__ inline int entries64(const BandDev &b, const Tile &tl, int t, double rc, const GridF &,
                                Entries64 &E, double) {
    const ImgScalars &sc = b.sc[tl.img];
    const size_t base = (size_t)tl.img * b.n;
    const double4_32a *off = (const double4_32a *)b.slot_off + base;
    const int *nslot = b.nbr_slot + base * MAXN_TERSOFF;
    const int *ncode = b.nbr_code + base * MAXN_TERSOFF;
    const int ne = b.nbr_cnt[base + t] & NBR_COUNT;
    int b0, b1, b2;
    unpack_bin(b.slot_bin[base + t], b0, b1, b2);
    const double4_32a oi = off[t];
    int cnt = 0;
    for (int e = 0; e < ne; ++e) {
        const double4_32a oj = off[nslot[ent(e, t, b.n)]];
        int d[3], w[3];
        ters_code(ncode[ent(e, t, b.n)], b0, b1, b2, sc.nb, d, w);
        double v[3] = {oj.x - oi.x, oj.y - oi.y, oj.z - oi.z};
        for (int c = 0; c < 3; ++c) {
            v[c] += f2d(d[0] * sc.bvf[c] + d[1] * sc.bvf[3 + c] + d[2] * sc.bvf[6 + c]);
            if (w[0] | w[1] | w[2])
                v[c] += f2d((float)w[0]) * sc.dh[c] + f2d((float)w[1]) * sc.dh[3 + c] +
                        f2d((float)w[2]) * sc.dh[6 + c];
        }
        cnt += add_entry(E, cnt, v[0], v[1], v[2], rc * rc);
    }
    return cnt;
}

// FP64 site energies.  Bound by the FP64 pipe: angular terms run over unordered
// pairs (symmetric in j, k), constants derived on the host, reciprocals by
// Newton steps (98,304 carbon atoms: 152 us; 282 us with ordered pairs,
// divisions and FP64 conversions of every coordinate).
template <typename T>
__global__ void __launch_bounds__(TILE) k_energy64(const Tile *tiles, BandDev *bands) {
    Tile tl = tiles[blockIdx.x];
    BandDev &b = bands[tl.band];
    const BandParams *bp = b.bp;
    __shared__ GridF G;
    __shared__ TP<double> q;
    if (sizeof(T) == 4) grid_stage(G, b, tl.img);
    stage_copy(&q, &bp->tpd);
    __syncthreads();
    const int t = tile_atom(b, tl);
    double U = 0.0;
    if (t < b.n) {
        Entries64 E;
        if (bp->kind == KIND_TERSOFF) {
            const int cnt = entries64(b, tl, t, q.R + q.D, G, E, T());
            double fc[MAXN_TERSOFF], zeta[MAXN_TERSOFF];
            for (int k = 0; k < cnt; ++k) {
                const double s = E.r[k] - q.R;
                fc[k] = 1.0;
                if (s > -q.D) {
                    const double sn = s < q.D ? sin_quarter64(q.pi_4D * (q.D - s)) : 0.0;
                    fc[k] = sn * sn;
                }
                zeta[k] = 0.0;
            }
            for (int j = 1; j < cnt; ++j) {
                double zj = 0.0;
                for (int k = 0; k < j; ++k) {
                    const double u = q.h - (E.x[j] * E.x[k] + E.y[j] * E.y[k] + E.z[j] * E.z[k]);
                    const double u2 = u * u;
                    const double g = fma(q.c2d2 * u2, rcp64_pos(q.d2 + u2), 1.0);
                    zj = fma(fc[k], g, zj);
                    zeta[k] = fma(fc[j], g, zeta[k]);
                }
                zeta[j] += zj;
            }
            for (int j = 0; j < cnt; ++j) {
                if (fc[j] == 0.0) continue;  // beyond R + D
                const double bz = q.beta * zeta[j];
                const double bij = bz > 0.0 ? bond_order_x(exp(q.n * log(bz)), q.inv2n, q.xs) : 1.0;
                U += 0.5 * fc[j] * (q.A * exp(-q.l1 * E.r[j]) - bij * q.B * exp(-q.l2 * E.r[j]));
            }
        } else {
            // NEP-style site energy (descriptors and network as in the force
            // kernel)
            const double rc = bp->pot[0], irc = rcp64_pos(rc);
            const int cnt = entries64(b, tl, t, rc, G, E, T());
            const double *w = b.nep_w;
            double qd[NEP_ND], gA[MAXN_TERSOFF][NEP_NA];
            for (int d = 0; d < NEP_ND; ++d) qd[d] = 0.0;
            for (int j = 0; j < cnt; ++j) {
                const double rr = E.r[j] * irc;
                const double fcj = 0.5 * (1.0 + cospi(rr));
                const double x = 2.0 * (rr - 1.0) * (rr - 1.0) - 1.0;
                double f[NEP_K], t0 = 1.0, t1 = x;
                f[0] = fcj;
                f[1] = 0.5 * (x + 1.0) * fcj;
                for (int k = 2; k < NEP_K; ++k) {
                    const double t2 = 2.0 * x * t1 - t0;
                    f[k] = 0.5 * (t2 + 1.0) * fcj;
                    t0 = t1;
                    t1 = t2;
                }
                for (int m = 0; m < NEP_NR; ++m)
                    for (int k = 0; k < NEP_K; ++k) qd[m] += w[NEP_OCR + m * NEP_K + k] * f[k];
                for (int m = 0; m < NEP_NA; ++m) {
                    gA[j][m] = 0.0;
                    for (int k = 0; k < NEP_K; ++k) gA[j][m] += w[NEP_OCA + m * NEP_K + k] * f[k];
                }
            }
            for (int j = 0; j < cnt; ++j) {
                for (int m = 0; m < NEP_NA; ++m)  // k = j: P_l(1) = 1
                    for (int l = 0; l < NEP_L; ++l) qd[NEP_NR + m * NEP_L + l] += gA[j][m] * gA[j][m];
                for (int k = 0; k < j; ++k) {
                    const double c = E.x[j] * E.x[k] + E.y[j] * E.y[k] + E.z[j] * E.z[k];
                    const double P[4] = {c, 1.5 * c * c - 0.5, (2.5 * c * c - 1.5) * c,
                                         (4.375 * c * c - 3.75) * c * c + 0.375};
                    for (int m = 0; m < NEP_NA; ++m) {
                        const double gg = 2.0 * gA[j][m] * gA[k][m];
                        for (int l = 0; l < NEP_L; ++l) qd[NEP_NR + m * NEP_L + l] += gg * P[l];
                    }
                }
            }
            double Ui = -w[NEP_OB1];
            for (int h = 0; h < NEP_H; ++h) {
                double a = -w[NEP_OB0 + h];
                for (int d = 0; d < NEP_ND; ++d) a += w[NEP_OW0 + h * NEP_ND + d] * qd[d];
                Ui += w[NEP_OW1 + h] * tanh(a);
            }
            U += Ui;
        }
    }
    double acc[1] = {U};
    double tot[1];
    block_sum<1>(acc, tot);
    if (threadIdx.x == 0) b.atom_part[((size_t)tl.img * b.atpi + tl.t) * NPART] = tot[0];
}

// one block per image: E64 = sum of the tile energies (+ P Omega)
__global__ void k_energy_finalize(const ImgRef *imgs, BandDev *bands) {
    ImgRef r = imgs[blockIdx.x];
    BandDev &b = bands[r.band];
    const double *part = b.atom_part + (size_t)r.img * b.atpi * NPART;
    double v[1] = {0.0}, s[1];
    for (int t = threadIdx.x; t < b.atpi; t += blockDim.x) v[0] += part[(size_t)t * NPART];
    block_sum_any<1>(v, s);
    if (threadIdx.x == 0) b.sc[r.img].E64 = s[0] + b.bp->pressure * b.sc[r.img].omega;
}

template <typename T>
void launch_energy64(const Tile *tiles, int ntiles, BandDev *bands, cudaStream_t s) {
    if (ntiles <= 0) return;
    k_energy64<T><<<ntiles, TILE, 0, s>>>(tiles, bands);
}
void launch_energy_finalize(const ImgRef *imgs, int nimg, BandDev *bands, cudaStream_t s) {
    if (nimg <= 0) return;
    k_energy_finalize<<<nimg, RED_THREADS, 0, s>>>(imgs, bands);
}
template void launch_energy64<float>(const Tile *, int, BandDev *, cudaStream_t);
template void launch_energy64<double>(const Tile *, int, BandDev *, cudaStream_t);

}  // namespace cfneb
