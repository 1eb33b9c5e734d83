// propagate_f64.cu -- all-FP64 mode (PAMD_PREC_FP64): the same method with
// every quantity in binary64 on the GPU, as a precision reference for the
// mixed FP32/FP64 kernels.
//
// Layout: replica state [R][6][Np] doubles.  GB300 issues two FP64 operations
// per clock and SM, one warp instruction in 16 cycles, so the kernel is bound
// by the number of FP64 warp instructions, and everything here serves that:
//   * L lanes of a warp share a replica, lane g owns atoms [gB, gB + B), and
//     the warp holds 32 / L replicas (the shape of the mixed kernels: 2 x 15
//     lanes x 5 atoms at 75 atoms, 30 of 32 lanes busy);
//   * Newton's third law over the half ring of lane blocks: tile t pairs block
//     g with block (g + t) mod L; the partner atoms' forces are summed in
//     registers and handed to their owner by shuffles after the tile;
//   * what a pair's types decide, 48 eps sigma^12, 24 eps sigma^6 and k_e q q
//     with the 1-4 factors, is read from a table made on the host ([tile][b]
//     [a][lane], L2-resident), with a bit for each pair that does not count
//     (excluded, padding, the idle half of the antipodal tile);
//   * one reciprocal square root per pair and no division; bonded terms with
//     one reciprocal per length and dihedral forces from cos and sin of the
//     torsion by multiple-angle formulas, without inverse or direct
//     trigonometric functions;
//   * one warp per block, so that a population spreads evenly over the SMs,
//     and a shape chosen by the instructions of the fullest SM
//     (choose_lanes_f64), so that a small population uses more lanes per
//     replica.
// 24 FP64 operations per pair instead of about 80 for each of both ordered
// pairs.  75 atoms, R = 2048: 0.44 ms per step with the FP64 pipe
// full (7535 FP64 instructions per warp and step); one warp per replica over all N^2
// ordered pairs with two square roots and three divisions each took 2.4 ms.
// Bonded forces go to per-atom shared-memory accumulators with atomicAdd.
// Noise, init and resampling use the same Philox counters as the mixed path,
// Box-Muller in double.
#include <math.h>

#include "pamd_device.cuh"
#include "pamd_internal.h"

namespace pamd {

namespace {

__device__ __forceinline__ double u23d(uint32_t u) { return ((double)(u >> 9) + 0.5) * 0x1p-23; }

__device__ __forceinline__ void normal3d(unsigned long long seed, uint32_t atom, uint32_t slot,
                                         uint32_t step, uint32_t purpose, double z[3]) {
    const uint4 o = philox4x32_10(make_uint4(atom, slot, step, purpose), seed_key(seed));
    const double r0 = sqrt(-2.0 * log(u23d(o.x)));
    const double r1 = sqrt(-2.0 * log(u23d(o.z)));
    double sn, cs;
    sincospi(2.0 * u23d(o.y), &sn, &cs);  // 2 u is exact
    z[0] = r0 * cs;
    z[1] = r0 * sn;
    z[2] = r1 * cospi(2.0 * u23d(o.w));
}

struct D3 {
    double x, y, z;
};
__device__ __forceinline__ D3 dsub(D3 a, D3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ double ddot(D3 a, D3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ D3 dcross(D3 a, D3 b) {
    return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}

// Positions (and bonded forces) of one replica in shared memory: three
// coordinate planes of L blocks of B atoms at an odd block stride.
template <int B>
struct Slots {
    double* p;
    int plane;
    __device__ __forceinline__ int at(int i) const { return (i / B) * (B | 1) + i % B; }
    __device__ __forceinline__ D3 get(int i) const {
        const int q = at(i);
        return {p[q], p[plane + q], p[2 * plane + q]};
    }
    __device__ __forceinline__ void add(int i, bool on, double fx, double fy, double fz) const {
        if (on) {
            const int q = at(i);
            atomicAdd(&p[q], fx);
            atomicAdd(&p[plane + q], fy);
            atomicAdd(&p[2 * plane + q], fz);
        }
        __syncwarp();
    }
};

// Bonded forces, the L lanes of a replica striding over each list.  Every
// lane of the warp runs every trip, past the end of a list on its last term
// with the additions switched off: with trip counts that differ between lanes
// the replicas of a warp come apart and stay apart through the pair loops
// (17.5 of 32 lanes active, a block of 4 steps took 4.2 ms instead of 2.5).
template <int B>
__device__ __forceinline__ void bonded_forces_f64(const TopoF64& t, const Slots<B> pos, const Slots<B> frc, int g,
                                                  int L, bool lane_on) {
    for (int b0 = 0; b0 < t.n_bonds; b0 += L) {
        const bool on = lane_on && b0 + g < t.n_bonds;
        const int b = min(b0 + g, t.n_bonds - 1);
        const int i = t.bond[2 * b], j = t.bond[2 * b + 1];
        const D3 d = dsub(pos.get(i), pos.get(j));
        const double r0 = t.bond_p[2 * b], k = t.bond_p[2 * b + 1];
        const double w = (r0 == 0.0) ? k : k * (1.0 - r0 * rsqrt(ddot(d, d)));
        __syncwarp();
        frc.add(i, on, -w * d.x, -w * d.y, -w * d.z);
        frc.add(j, on, w * d.x, w * d.y, w * d.z);
    }
    for (int a0 = 0; a0 < t.n_angles; a0 += L) {
        const bool on = lane_on && a0 + g < t.n_angles;
        const int a = min(a0 + g, t.n_angles - 1);
        const int i = t.angle[3 * a], j = t.angle[3 * a + 1], k = t.angle[3 * a + 2];
        const D3 xj = pos.get(j), u = dsub(pos.get(i), xj), w = dsub(pos.get(k), xj), n = dcross(u, w);
        const double ss = ddot(n, n), is = rsqrt(ss), c = ddot(u, w);
        const double th = atan2(ss * is, c);
        __syncwarp();
        const double q = t.angle_p[2 * a + 1] * (th - t.angle_p[2 * a]) * is;
        const double cu = c / ddot(u, u), cw = c / ddot(w, w);
        const D3 fi = {q * (w.x - cu * u.x), q * (w.y - cu * u.y), q * (w.z - cu * u.z)};
        const D3 fk = {q * (u.x - cw * w.x), q * (u.y - cw * w.y), q * (u.z - cw * w.z)};
        frc.add(i, on, fi.x, fi.y, fi.z);
        frc.add(k, on, fk.x, fk.y, fk.z);
        frc.add(j, on, -fi.x - fk.x, -fi.y - fk.y, -fi.z - fk.z);
    }
    for (int h0 = 0; h0 < t.n_dihs; h0 += L) {
        const bool on = lane_on && h0 + g < t.n_dihs;
        const int h = min(h0 + g, t.n_dihs - 1);
        const int i = t.dih[4 * h], j = t.dih[4 * h + 1], k = t.dih[4 * h + 2], l = t.dih[4 * h + 3];
        const double kd = t.dih_p[4 * h];
        const int n = (int)t.dih_p[4 * h + 1];
        const D3 xj = pos.get(j), xk = pos.get(k);
        const D3 F = dsub(pos.get(i), xj), G = dsub(xj, xk), H = dsub(pos.get(l), xk);
        const D3 A = dcross(F, G), Bv = dcross(H, G);
        const double gg = ddot(G, G), ilg = rsqrt(gg), lg = gg * ilg;
        // cos and sin of the torsion: A.B and (B x A).G / |G| = -|G| F.B over their norm
        double c = ddot(A, Bv), sn = -lg * ddot(F, Bv);
        const double in = rsqrt(c * c + sn * sn);
        c *= in;
        sn *= in;
        double cn = c, snn = sn;
        const int n_max = __reduce_max_sync(0xffffffffu, n);
        for (int q = 1; q < n_max; ++q) {
            const double t2 = cn * c - snn * sn, t3 = snn * c + cn * sn;
            cn = q < n ? t2 : cn;
            snn = q < n ? t3 : snn;
        }
        const double dEdphi = -kd * n * (snn * t.dih_p[4 * h + 2] - cn * t.dih_p[4 * h + 3]);
        const double ra = 1.0 / ddot(A, A), rb = 1.0 / ddot(Bv, Bv);
        __syncwarp();
        const double ia = lg * ra, ib = lg * rb;
        const double pa = ddot(F, G) * ra * ilg, pb = ddot(H, G) * rb * ilg;
        frc.add(i, on, dEdphi * ia * A.x, dEdphi * ia * A.y, dEdphi * ia * A.z);
        frc.add(l, on, -dEdphi * ib * Bv.x, -dEdphi * ib * Bv.y, -dEdphi * ib * Bv.z);
        const double ja = -dEdphi * (ia + pa), jb = dEdphi * pb;
        const double ka = dEdphi * pa, kb = -dEdphi * (pb - ib);
        frc.add(j, on, ja * A.x + jb * Bv.x, ja * A.y + jb * Bv.y, ja * A.z + jb * Bv.z);
        frc.add(k, on, ka * A.x + kb * Bv.x, ka * A.y + kb * Bv.y, ka * A.z + kb * Bv.z);
    }
}

// This lane's share of the bonded energy.
template <int B>
__device__ __forceinline__ double bonded_energy_f64(const TopoF64& t, const Slots<B> pos, int g, int L) {
    double e = 0.0;
    for (int b = g; b < t.n_bonds; b += L) {
        const D3 d = dsub(pos.get(t.bond[2 * b]), pos.get(t.bond[2 * b + 1]));
        const double dr = sqrt(ddot(d, d)) - t.bond_p[2 * b];
        e += 0.5 * t.bond_p[2 * b + 1] * dr * dr;
    }
    for (int a = g; a < t.n_angles; a += L) {
        const D3 xj = pos.get(t.angle[3 * a + 1]);
        const D3 u = dsub(pos.get(t.angle[3 * a]), xj), w = dsub(pos.get(t.angle[3 * a + 2]), xj);
        const D3 n = dcross(u, w);
        const double dth = atan2(sqrt(ddot(n, n)), ddot(u, w)) - t.angle_p[2 * a];
        e += 0.5 * t.angle_p[2 * a + 1] * dth * dth;
    }
    for (int h = g; h < t.n_dihs; h += L) {
        const double nn = t.dih_p[4 * h + 1];
        const D3 xj = pos.get(t.dih[4 * h + 1]), xk = pos.get(t.dih[4 * h + 2]);
        const D3 F = dsub(pos.get(t.dih[4 * h]), xj), G = dsub(xj, xk), H = dsub(pos.get(t.dih[4 * h + 3]), xk);
        const D3 A = dcross(F, G), Bv = dcross(H, G);
        const double phi = atan2(ddot(dcross(Bv, A), G) / sqrt(ddot(G, G)), ddot(A, Bv));
        e += t.dih_p[4 * h] * (1.0 + cos(nn * phi) * t.dih_p[4 * h + 2] + sin(nn * phi) * t.dih_p[4 * h + 3]);
    }
    return e;
}

// One nonbonded pair: d = x_i - x_j, c12 = 48 eps sigma^12, c6 = 24 eps
// sigma^6, qq = k_e q_i q_j.  FORCE returns w with force w d on i and -w d on
// j, else the energy.
template <bool FORCE>
__device__ __forceinline__ double nb_pair_f64(const D3 d, bool off, double c12, double c6, double qq) {
    double r2 = ddot(d, d);
    if (off) r2 = 1.0;  // a pair that does not count: its coefficients are zero
    const double ir = rsqrt(r2), ir2 = ir * ir, ir6 = ir2 * ir2 * ir2;
    if (FORCE) return fma(fma(c12, ir6, -c6), ir6, qq * ir) * ir2;
    return fma(fma(c12 * (1.0 / 12.0), ir6, c6 * (-1.0 / 6.0)), ir6, qq * ir);
}

// All nonbonded pairs of this lane's tiles: forces on its own atoms in f
// (FORCE), or its share of the energy (returned).  Every lane of the warp
// takes part; idle lanes mirror a busy one and their results go unused.
template <int B, bool FORCE>
__device__ __forceinline__ double nonbonded_f64(const double* __restrict__ tab,
                                                const unsigned long long* __restrict__ off, const double* pos, int plane, int stride,
                                                const D3 (&x)[B], D3 (&f)[B], int g, int L, int base) {
    double e = 0.0;
    const int TH = L / 2;
    const unsigned long long m0 = off[g];
#pragma unroll
    for (int a = 0; a < B; ++a)
#pragma unroll
        for (int b = a + 1; b < B; ++b) {
            const double* q = tab + (size_t)((b * B + a) * 3) * L + g;
            const D3 d = dsub(x[a], x[b]);
            const double w = nb_pair_f64<FORCE>(d, (m0 >> (b * B + a)) & 1ull, q[0], q[L], q[2 * L]);
            if (FORCE) {
                f[a].x += w * d.x; f[a].y += w * d.y; f[a].z += w * d.z;
                f[b].x -= w * d.x; f[b].y -= w * d.y; f[b].z -= w * d.z;
            } else {
                e += w;
            }
        }
    for (int t = 1; t <= TH; ++t) {
        const int J = g + t < L ? g + t : g + t - L;
        const double* pj = pos + J * stride;
        const double* tt = tab + (size_t)t * B * B * 3 * L + g;
        const unsigned long long mt = off[t * L + g];
        D3 pf[B];
#pragma unroll
        for (int b = 0; b < B; ++b) {
            const D3 xj = {pj[b], pj[plane + b], pj[2 * plane + b]};
            pf[b] = {0.0, 0.0, 0.0};
#pragma unroll
            for (int a = 0; a < B; ++a) {
                const double* q = tt + (size_t)((b * B + a) * 3) * L;
                const D3 d = dsub(x[a], xj);
                const double w = nb_pair_f64<FORCE>(d, (mt >> (b * B + a)) & 1ull, q[0], q[L], q[2 * L]);
                if (FORCE) {
                    f[a].x += w * d.x; f[a].y += w * d.y; f[a].z += w * d.z;
                    pf[b].x -= w * d.x; pf[b].y -= w * d.y; pf[b].z -= w * d.z;
                } else {
                    e += w;
                }
            }
        }
        if (FORCE) {  // block g receives what lane g - t summed for it
            const int from = base + (g >= t ? g - t : g - t + L);
#pragma unroll
            for (int b = 0; b < B; ++b) {
                f[b].x += __shfl_sync(0xffffffffu, pf[b].x, from);
                f[b].y += __shfl_sync(0xffffffffu, pf[b].y, from);
                f[b].z += __shfl_sync(0xffffffffu, pf[b].z, from);
            }
        }
    }
    return e;
}

// Dynamic shared memory of one warp, in doubles: per replica positions and
// bonded forces, then per lane the velocities [3 B], dt / 2m [B] and the noise
// scale [B], and the sums' scratch.
template <int B>
__global__ void __launch_bounds__(32) propagate_f64_kernel(PropF64Params p) {
    extern __shared__ double smem_d[];
    const TopoF64& t = p.top;
    const int N = t.n_atoms, Np = p.n_pad, L = t.lanes, G = 32 / L;
    const int lane = threadIdx.x, grp_raw = lane / L, grp = grp_raw < G ? grp_raw : 0;
    const int g = grp_raw < G ? lane - grp * L : lane - G * L;  // idle lanes mirror lanes of the first group
    const int base = grp * L;
    const int stride = B | 1, plane = L * stride;
    const Slots<B> pos{smem_d + (size_t)grp * 6 * plane, plane};
    const Slots<B> frc{pos.p + 3 * plane, plane};
    double* vel = smem_d + (size_t)G * 6 * plane + lane;  // component c of atom a: vel[32 (c B + a)]
    double* hmv = vel + 32 * 3 * B;  // dt / 2m of atom a: hmv[32 a]
    double* sdv = hmv + 32 * B;      // noise scale
    double* scratch = smem_d + (size_t)G * 6 * plane + 32 * 5 * B;
    const uint32_t step_base = (p.dev_counters ? p.dev_counters[0] : 0u) + p.step0;
    const double c1 = exp(-p.gamma * p.dt), c2kT = sqrt((1.0 - c1 * c1) * kBoltzmann * p.T);
    const double hdt = 0.5 * p.dt;
#pragma unroll
    for (int a = 0; a < B; ++a) {
        const double im = g * B + a < N ? t.inv_mass[g * B + a] : 0.0;
        hmv[32 * a] = hdt * im;
        sdv[32 * a] = c2kT * sqrt(im);
    }
    for (long long k0 = (long long)blockIdx.x * G; k0 < p.R; k0 += (long long)gridDim.x * G) {
        const bool live = grp_raw < G && k0 + grp < p.R;
        const long long k = k0 + grp < p.R ? k0 + grp : p.R - 1;  // a missing replica repeats the last one
        double* st = p.state + (size_t)k * 6 * Np;
        D3 x[B], f[B];
#pragma unroll
        for (int a = 0; a < B; ++a) {
            const int i = g * B + a;
            const bool real = i < N;
            x[a] = {real ? st[i] : 0.0, real ? st[Np + i] : 0.0, real ? st[2 * Np + i] : 0.0};
#pragma unroll
            for (int c = 0; c < 3; ++c) vel[32 * (c * B + a)] = real ? st[(3 + c) * Np + i] : 0.0;
        }
        // s = -1 evaluates the forces of the incoming state
        for (int s = -1; s < p.theta; ++s) {
            if (s >= 0) {
                const uint32_t step = step_base + (uint32_t)s;
#pragma unroll
                for (int a = 0; a < B; ++a) {
                    const int i = g * B + a;
                    if (i >= N) continue;
                    const double sd = sdv[32 * a], hm = hmv[32 * a];
                    double z[3];
                    normal3d(p.seed, (uint32_t)i, (uint32_t)k, step, p.purpose_mol, z);
                    const double fa[3] = {f[a].x, f[a].y, f[a].z};
                    double xa[3] = {x[a].x, x[a].y, x[a].z};
#pragma unroll
                    for (int c = 0; c < 3; ++c) {
                        double v = vel[32 * (c * B + a)];
                        v += hm * fa[c];
                        xa[c] += hdt * v;
                        v = c1 * v + sd * z[c];
                        xa[c] += hdt * v;
                        vel[32 * (c * B + a)] = v;
                    }
                    x[a] = {xa[0], xa[1], xa[2]};
                }
            }
            __syncwarp();  // the previous step's readers of pos and frc are done
            if (grp_raw < G) {
#pragma unroll
                for (int a = 0; a < B; ++a) {
                    const int q = g * stride + a;
                    pos.p[q] = x[a].x; pos.p[plane + q] = x[a].y; pos.p[2 * plane + q] = x[a].z;
                    frc.p[q] = 0.0; frc.p[plane + q] = 0.0; frc.p[2 * plane + q] = 0.0;
                }
            }
            __syncwarp();
            bonded_forces_f64(t, pos, frc, g, L, grp_raw < G);
#pragma unroll
            for (int a = 0; a < B; ++a) f[a] = {0.0, 0.0, 0.0};
            __syncwarp();
            nonbonded_f64<B, true>(t.tab, t.off, pos.p, plane, stride, x, f, g, L, base);
#pragma unroll
            for (int a = 0; a < B; ++a) {
                const int i = g * B + a, q = g * stride + a;
                f[a].x += frc.p[q]; f[a].y += frc.p[plane + q]; f[a].z += frc.p[2 * plane + q];
                if (s < 0 || i >= N) continue;
                const double hm = hmv[32 * a];
                vel[32 * a] += hm * f[a].x;
                vel[32 * (B + a)] += hm * f[a].y;
                vel[32 * (2 * B + a)] += hm * f[a].z;
            }
        }
        // energy and per-replica observables
        double e = nonbonded_f64<B, false>(t.tab, t.off, pos.p, plane, stride, x, f, g, L, base);
        if (grp_raw < G) e += bonded_energy_f64(t, pos, g, L);
        double ek = 0.0, cx = 0.0, cy = 0.0, cz = 0.0;
#pragma unroll
        for (int a = 0; a < B; ++a) {
            const int i = g * B + a;
            if (i >= N) continue;
            const double vx = vel[32 * a], vy = vel[32 * (B + a)], vz = vel[32 * (2 * B + a)];
            if (live && p.theta > 0) {
                st[i] = x[a].x; st[Np + i] = x[a].y; st[2 * Np + i] = x[a].z;
                st[3 * Np + i] = vx; st[4 * Np + i] = vy; st[5 * Np + i] = vz;
            }
            if (live && p.fout) {
                double* fo = p.fout + (size_t)k * 3 * Np;
                fo[i] = f[a].x; fo[Np + i] = f[a].y; fo[2 * Np + i] = f[a].z;
            }
            ek += 0.5 * (1.0 / t.inv_mass[i]) * (vx * vx + vy * vy + vz * vz);
            cx += x[a].x; cy += x[a].y; cz += x[a].z;
        }
        // sum over the replica's lanes, in lane order
        auto total = [&](double v) {
            __syncwarp();
            scratch[lane] = v;
            __syncwarp();
            double s = 0.0;
            for (int q = 0; q < L; ++q) s += scratch[base + q];
            return s;
        };
        e = total(e);
        ek = total(ek);
        cx = total(cx) / N;
        cy = total(cy) / N;
        cz = total(cz) / N;
        double r2 = 0.0;
#pragma unroll
        for (int a = 0; a < B; ++a) {
            if (g * B + a >= N) continue;
            const double dx = x[a].x - cx, dy = x[a].y - cy, dz = x[a].z - cz;
            r2 += dx * dx + dy * dy + dz * dz;
        }
        r2 = total(r2);
        if (live && g == 0) {
            p.E[k] = e;
            p.ke[k] = ek;
            p.rg[k] = sqrt(r2 / N);
            if (!isfinite(e) && atomicCAS(&p.status[0], 0, PAMD_ENONFINITE) == 0) p.status[1] = (int)k;
        }
        __syncwarp();
    }
}

__global__ void init_f64_kernel(double* state, double* E, int32_t* fam, const double* x0,
                                const double* inv_mass, long long R, int N, int Np, double kT0,
                                unsigned long long seed, uint32_t purpose) {
    const long long total = R * (long long)Np;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const long long k = t / Np;
        const int i = (int)(t - k * Np);
        double* st = state + (size_t)k * 6 * Np;
        if (i < N) {
            double z[3];
            normal3d(seed, (uint32_t)i, (uint32_t)k, 0u, purpose, z);
            const double sdv = sqrt(kT0 * inv_mass[i]);
            st[i] = x0[i];
            st[Np + i] = x0[Np + i];
            st[2 * Np + i] = x0[2 * Np + i];
            st[3 * Np + i] = sdv * z[0];
            st[4 * Np + i] = sdv * z[1];
            st[5 * Np + i] = sdv * z[2];
        } else {
#pragma unroll
            for (int c = 0; c < 6; ++c) st[c * Np + i] = 0.0;
        }
        if (i == 0) {
            fam[k] = (int32_t)k;
            E[k] = 0.0;
        }
    }
}

// One warp per new slot k, ancestor by binary search of the inclusive counts;
// positions recentred on the centre of mass, velocities scaled.
__global__ void gather_f64_kernel(const double* __restrict__ st_in, double* __restrict__ st_out,
                                  const double* E_in, double* E_out, const int32_t* fam_in,
                                  int32_t* fam_out, double* ke_out, double* rg_out,
                                  const int32_t* incl, const double* inv_mass, long long R, int N,
                                  int Np, double vscale) {
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long k = warp; k < R; k += nwarps) {
        long long lo = 0, hi = R;
        while (lo < hi) {
            const long long mid = lo + ((hi - lo) >> 1);
            if (incl[mid] > k) hi = mid;
            else lo = mid + 1;
        }
        const long long j = lo < R ? lo : R - 1;
        const double* src = st_in + (size_t)j * 6 * Np;
        double* dst = st_out + (size_t)k * 6 * Np;
        double m = 0.0, sx = 0.0, sy = 0.0, sz = 0.0;
        for (int i = lane; i < N; i += 32) {
            const double mi = 1.0 / inv_mass[i];
            m += mi;
            sx += mi * src[i];
            sy += mi * src[Np + i];
            sz += mi * src[2 * Np + i];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            m += __shfl_xor_sync(0xffffffffu, m, o);
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
            sy += __shfl_xor_sync(0xffffffffu, sy, o);
            sz += __shfl_xor_sync(0xffffffffu, sz, o);
        }
        const double cx = sx / m, cy = sy / m, cz = sz / m;
        double mv2 = 0.0, ux = 0.0, uy = 0.0, uz = 0.0, u2 = 0.0;
        for (int i = lane; i < Np; i += 32) {
            if (i < N) {
                const double x = src[i] - cx, y = src[Np + i] - cy, z = src[2 * Np + i] - cz;
                const double vx = vscale * src[3 * Np + i], vy = vscale * src[4 * Np + i],
                             vz = vscale * src[5 * Np + i];
                dst[i] = x; dst[Np + i] = y; dst[2 * Np + i] = z;
                dst[3 * Np + i] = vx; dst[4 * Np + i] = vy; dst[5 * Np + i] = vz;
                mv2 += (vx * vx + vy * vy + vz * vz) / inv_mass[i];
                ux += x; uy += y; uz += z;
                u2 += x * x + y * y + z * z;
            } else {
#pragma unroll
                for (int c = 0; c < 6; ++c) dst[c * Np + i] = 0.0;
            }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            mv2 += __shfl_xor_sync(0xffffffffu, mv2, o);
            ux += __shfl_xor_sync(0xffffffffu, ux, o);
            uy += __shfl_xor_sync(0xffffffffu, uy, o);
            uz += __shfl_xor_sync(0xffffffffu, uz, o);
            u2 += __shfl_xor_sync(0xffffffffu, u2, o);
        }
        if (lane == 0) {
            E_out[k] = E_in[j];
            fam_out[k] = fam_in[j];
            ke_out[k] = 0.5 * mv2;
            const double mx = ux / N, my = uy / N, mz = uz / N;
            rg_out[k] = sqrt(fmax(u2 / N - (mx * mx + my * my + mz * mz), 0.0));
        }
    }
}

}  // namespace

cudaError_t launch_propagate_f64(pamd_ctx* c, double* state, double* E, double* ke, double* rg,
                                 int theta, double dt, double T, const uint32_t* dev_ctr,
                                 uint32_t step0, double* fout) {
    PropF64Params p{};
    p.state = state;
    p.E = E;
    p.ke = ke;
    p.rg = rg;
    p.fout = fout;
    p.status = &c->b.scal->status;
    p.dev_counters = dev_ctr;
    p.top = c->top64;
    p.n_pad = c->Np;
    p.R = c->R;
    p.theta = theta;
    p.dt = dt;
    p.T = T;
    p.gamma = c->gamma;
    p.seed = c->seed;
    p.step0 = step0;
    p.purpose_mol = kPurposeNoise | ((uint32_t)c->mol << 8);
    const int L = p.top.lanes, B = p.top.per_lane, G = 32 / L;
    const size_t smem = sizeof(double) * ((size_t)G * 6 * L * (B | 1) + 32 * 5 * (size_t)B + 32);
    const long long warps = (c->R + G - 1) / G;
    const int grid = (int)(warps < (long long)c->num_sms * 32 ? warps : (long long)c->num_sms * 32);
    cudaError_t e = cudaSuccess;
    switch (B) {
#define PAMD_F64_CASE(A)                                                              \
    case A:                                                                           \
        e = ensure_dyn_smem((const void*)propagate_f64_kernel<A>, smem);              \
        if (e == cudaSuccess) propagate_f64_kernel<A><<<grid, 32, smem, c->stream>>>(p); \
        break;
        PAMD_F64_CASE(1) PAMD_F64_CASE(2) PAMD_F64_CASE(3) PAMD_F64_CASE(4)
        PAMD_F64_CASE(5) PAMD_F64_CASE(6) PAMD_F64_CASE(7) PAMD_F64_CASE(8)
#undef PAMD_F64_CASE
        default: return cudaErrorInvalidValue;
    }
    c->launches += 1;
    if (e != cudaSuccess) return e;
    return cudaGetLastError();
}

cudaError_t launch_init_f64(pamd_ctx* c, double T0) {
    const long long total = c->R * c->Np;
    long long g = (total + 255) / 256;
    if (g > (long long)c->num_sms * 16) g = (long long)c->num_sms * 16;
    init_f64_kernel<<<(int)g, 256, 0, c->stream>>>(
        reinterpret_cast<double*>(c->b.state), c->b.E, c->b.fam, c->top64.x0, c->top64.inv_mass,
        c->R, c->N, c->Np, kBoltzmann * T0, c->seed, kPurposeInit | ((uint32_t)c->mol << 8));
    c->launches += 1;
    return cudaGetLastError();
}

cudaError_t launch_gather_f64(pamd_ctx* c, const double* src, double* dst, const double* Ein,
                              double* Eout, const int32_t* fin, int32_t* fout, double vscale) {
    long long g = (c->R * 32 + 255) / 256;
    if (g > (long long)c->num_sms * 32) g = (long long)c->num_sms * 32;
    gather_f64_kernel<<<(int)g, 256, 0, c->stream>>>(src, dst, Ein, Eout, fin, fout, c->b.ke,
                                                       c->b.rg, c->b.cnt_incl, c->top64.inv_mass,
                                                       c->R, c->N, c->Np, vscale);
    c->launches += 1;
    return cudaGetLastError();
}

}  // namespace pamd
