// state_dev.cuh — device bodies of the FP64 prediction and of the pose
// matrices, shared by the single-stream kernels (state.cu) and the batched
// serving kernels (serve_kernels.cu).
//
// The FP64 prediction step (App. E.1 transition with the
// linearisation of App. E.1, Eq. statepropagation, App. E.2 split into the
// pose prior and the velocity conditional), on one block.
//
// Controls from the IMU window (reading R13): u_lin = R_mid mean(acc) + g,
// R_mid = Exp(w_m dt / 2) R; u_ang = (R_end w_end - w_prev) / dt with w_end
// the least-squares line through the gyro samples at the last sample time,
// R_end = Exp(w_m dt) R, w_m = R mean(gyro).  Velocity integration reads the
// printed (dt)^2 as dt (R12).  Error state (dt, dtheta, dv, dw) with the
// rotation error on the left (R14): A = diag(I, Exp(w dt)),
// B = diag(dt I, J_l(w dt) dt), F = [[A, B], [0, I]],
// Sigma' = F Sigma F^T + [[B Qv B^T + Qp, B Qv], [Qv B^T, Qv]].
// The kernel also starts the Gauss-Newton iterate at the prior mean.
#pragma once

#include "kernels.h"
#include "linalg64.cuh"
#include "prism_dev.cuh"

#include <cstddef>

namespace prism {

// v[0 .. N - 1] summed over the warp (N = 4 or 8): the sum of value k in the
// lanes l with l >> (N == 8 ? 2 : 3) == k (mod N), by the additions of a
// shuffle tree for each value (offsets 16, 8, 4, 2, 1), most of them shared:
// N - 1 + 5 - log2 N instead of 5 N FP64 additions.
template <int N>
__device__ __forceinline__ double warp_reduce_scatter64(double (&v)[N]) {
    const int lane = threadIdx.x & 31;
    int o = 16;
#pragma unroll
    for (int w = N / 2; w >= 1; w >>= 1, o >>= 1) {
        const bool upper = (lane & o) != 0;
#pragma unroll
        for (int i = 0; i < w; ++i) {
            const double send = sel64(upper, v[i], v[i + w]), keep = sel64(upper, v[i + w], v[i]);
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    }
    for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    return v[0];
}

// Doubles as unsigned integers in the same order, and back.
__device__ __forceinline__ unsigned long long ordered_bits(double d) {
    const long long b = __double_as_longlong(d);
    return (unsigned long long)(b < 0 ? ~b : b ^ (long long)0x8000000000000000ull);
}
__device__ __forceinline__ double from_ordered(unsigned long long u) {
    const long long b = (long long)u;
    return __longlong_as_double(b < 0 ? b ^ (long long)0x8000000000000000ull : ~b);
}

// The prediction on one block of 256 threads.  PREP = PREP_REL or
// PREP_REL_NEXT: also what prep_mats_warp derives for PREP_REL (the
// Gauss-Newton start matrices of the new prior, whose iterate xi = 0 makes
// J_l = I), against the anchor's pose or the state mean's; PREP_NONE: not.
//
// What bounds it: FP64 instructions, ~64 cycles each on one SM sub-partition
// whatever lanes are active, and the barriers between their chains.  So the
// products keep to the non-zero entries of F = [[A, B], [0, I]] (at most six of
// twelve in a row, one FMA a row of positions, none a row of velocities), the
// independent chains (IMU statistics, quaternions and rotation, reciprocals,
// noise terms, start matrices) run on warps of different sub-partitions, and
// the window's sums share their shuffle trees: 21 us alone with cold caches and 33
// IMU rows (35 with dense 12x12 products, five shuffles a sum and one warp's
// Cholesky with reciprocal square roots), 14.7 us a call in a loop of predictions
// with their uploads (23.4).  The warp index is read from lane 0 so that the compiler knows the
// branches on it to be warp-uniform: it otherwise takes every shuffle after
// the first loop for a divergent one (~500 cycles each instead of 25; the
// IMU statistics alone 16,800 cycles instead of 5,000).  The skipped products are by zeros: a covariance
// with an entry that is not finite, which they turned into NaN everywhere, is
// marked instead (bad) and rejected as before.
constexpr int PREP_NONE = -1;

template <int PREP>
__device__ __forceinline__ void predict_block(const KParams& P, DevState* dev, const double* __restrict__ imu,
                                              int n, double dt) {
    __shared__ double X[13];             // the state: t, q, v, w
    __shared__ double Cv[144], T1[144], Sig[144];
    __shared__ double R0[9], qm[4];      // of the normalised q
    __shared__ double E[18];             // Rw = Exp(w dt), Jd = J_l(w dt) dt
    __shared__ double qv[2];             // velocity noise variances, translation / rotation
    __shared__ double nz[20];            // noise: 0..8 rotation block, 9 position diagonal, 10..18 Jd qv, 19 dt qv
    __shared__ double sums[8], fit[4];   // mean t, acc (3), gyro (3), t_end; sum dt^2, sum dt dgyro (3)
    __shared__ double gend[3], wd[3], inv_dt, Me[18];
    __shared__ double pose[7], anchor[7], Ra[9];
    __shared__ double Prec[36], Dm[36], W[36], LC[36];
    __shared__ int ok;
    const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
    const double* state = reinterpret_cast<const double*>(reinterpret_cast<const char*>(dev) + offsetof(DevState, t));
    if (tid == 0) dev->flags = 0;   // a new step: only its own kernels raise flags
    bool bad = false;
    if (warp == 0) {
        // IMU window statistics: lane l takes samples l, l + 32, ...; the
        // reduction order is fixed, so the result is deterministic.
        const double inv_n = n > 0 ? 1.0 / n : 0.0;
        double a[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        unsigned long long te = ordered_bits(-1e300);
        for (int i0 = 0; i0 < n; i0 += 32) {
            const bool in = i0 + lane < n;
            const double* row = imu + 7 * (in ? i0 + lane : 0);
            double x[7];
            for (int c = 0; c < 7; ++c) x[c] = row[c];
            for (int c = 0; c < 7; ++c) a[c] = sel64(in, a[c] + x[c], a[c]);
            const unsigned long long k = ordered_bits(x[0]);
            te = in && k > te ? k : te;
        }
        const double mean = warp_reduce_scatter64<8>(a) * inv_n;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const unsigned long long k = __shfl_xor_sync(0xffffffffu, te, o);
            te = k > te ? k : te;
        }
        if ((lane & 3) == 0) sums[lane >> 2] = sel64(lane == 28, from_ordered(te), mean);
        __syncwarp();
        const double m0 = sums[0], m4[3] = {sums[4], sums[5], sums[6]};
        double f[4] = {0, 0, 0, 0};
        for (int i0 = 0; i0 < n; i0 += 32) {
            const bool in = i0 + lane < n;
            const double* row = imu + 7 * (in ? i0 + lane : 0);
            const double d = row[0] - m0;
            f[0] = sel64(in, fma(d, d, f[0]), f[0]);
            for (int c = 0; c < 3; ++c) f[1 + c] = sel64(in, fma(d, row[4 + c] - m4[c], f[1 + c]), f[1 + c]);
        }
        const double fs = warp_reduce_scatter64<4>(f);
        if ((lane & 7) == 0) fit[lane >> 3] = fs;
    } else if (warp == 7) {   // the normalised orientation (every lane the same operations) and its rotation
        double q[4] = {dev->q[0], dev->q[1], dev->q[2], dev->q[3]};
        quat_normalise(q);
        const double Re = quat_R_entry_rn(q[0], q[1], q[2], q[3], lane < 9 ? lane : 0);
        if (lane < 9) R0[lane] = Re;
        else if (lane < 13) qm[lane - 9] = sel64(lane == 9, q[0], sel64(lane == 10, q[1], sel64(lane == 11, q[2], q[3])));
    } else {
        const int e = tid - 32;   // 0 .. 191
        if (e < 157) {
            const double v = state[e];
            if (e < 13) X[e] = v;
            else Cv[e - 13] = v;
            bad = e >= 13 && !isfinite(v);
        } else if (PREP != PREP_NONE && e < 164) {
            anchor[e - 157] = PREP == PREP_REL_NEXT ? state[e - 157] : dev->anchor_pose[e - 157];
        }
        if (warp == 6) {
            const double r = 1.0 / dt;
            if (lane == 31) inv_dt = r;
        }
        if (tid == 32) ok = 1;
    }
    bad = __syncthreads_or(bad) != 0;
    // The controls: Rmid and Rend on warp 0, the gyro line's end on warp 1
    if (n > 0) {
        if (warp == 0) {
            const double gyr[3] = {sums[4], sums[5], sums[6]};
            // wm = R gyr (lane a < 3), then to every lane
            const int ra = lane < 3 ? lane : 0;
            const double wml = fdot3(R0[3 * ra], gyr[0], R0[3 * ra + 1], gyr[1], R0[3 * ra + 2], gyr[2]);
            // Rh = Exp(dt wm / 2) entries on lanes 0..8, Rf = Exp(dt wm) on lanes 9..17
            const bool hf = lane < 9;
            const int e = lane < 9 ? lane : (lane < 18 ? lane - 9 : 0), ei = e / 3, ej = e % 3;
            const double f = sel64(hf, 0.5 * dt, dt);
            double vrot[3];
            for (int a = 0; a < 3; ++a) vrot[a] = f * __shfl_sync(0xffffffffu, wml, a);
            const double Ee = so3_exp_jl_entry(vrot, true, ei, ej);
            // Rmid = Rh R on lanes 0..8, Rend = Rf R on lanes 9..17 (entry (i, j) a fdot3 over k)
            const int rb = hf ? 3 * ei : 9 + 3 * ei;
            const double m = fdot3(__shfl_sync(0xffffffffu, Ee, rb), R0[ej], __shfl_sync(0xffffffffu, Ee, rb + 1), R0[3 + ej],
                                   __shfl_sync(0xffffffffu, Ee, rb + 2), R0[6 + ej]);
            if (lane < 18) Me[lane] = m;
        } else if (warp == 1) {
            const double slope_scale = fit[0] > 0.0 ? (sums[7] - sums[0]) / fit[0] : 0.0;
            const int a = lane < 3 ? lane : 0;
            const double g = fma(fit[1 + a], slope_scale, sums[4 + a]);
            if (lane < 3) gend[lane] = g;
        }
    }
    if (warp == 2) {   // meanwhile: the noise variances, and the anchor's rotation
        const double s = P.sigma_vel[lane & 1];
        if (lane < 2) qv[lane] = s * s;
        if (PREP != PREP_NONE) {
            const double r = quat_R_entry_rn(anchor[3], anchor[4], anchor[5], anchor[6], lane < 9 ? lane : 0);
            if (lane < 9) Ra[lane] = r;
        }
    }
    __syncthreads();
    // The mean propagation on warp 0, one entry a lane
    if (warp == 0) {
        double u = 0.0;   // lanes 0..2: u_lin, lanes 3..5: u_ang (zero without IMU samples)
        if (n > 0) {
            // am = Rmid acc on lanes 0..2, we = Rend gend on lanes 3..5
            const bool lin = lane < 3;
            const int rr = lane < 3 ? lane : (lane < 6 ? lane - 3 : 0);
            const double* M = Me + (lin ? 0 : 9) + 3 * rr;
            const double* v = lin ? sums + 1 : gend;
            const double y = fdot3(M[0], v[0], M[1], v[1], M[2], v[2]);
            const double ul = y + sel64(lane == 2, -P.gravity, 0.0), ua = (y - X[10 + rr]) * inv_dt;
            u = sel64(lin, ul, ua);
        }
        // the new velocities (lanes 0..5) and position (lanes 0..2)
        const int l6 = lane < 6 ? lane : 0;
        const double vn = fma(u, dt, X[7 + l6]);
        const double vd = vn * dt;
        if (lane < 3) {
            const double p = fma(vn, dt, X[lane]);
            dev->pv[lane] = vn;
            dev->pt[lane] = p;
            pose[lane] = p;
        } else if (lane < 6) {
            dev->pw[lane - 3] = vn;
            wd[lane - 3] = vd;
        }
        double wdt[3];
        for (int a = 0; a < 3; ++a) wdt[a] = __shfl_sync(0xffffffffu, vd, 3 + a);
        // Rw = Exp(wdt) entries on lanes 0..8, J_l(wdt) dt on lanes 9..17
        const int e = lane < 9 ? lane : (lane < 18 ? lane - 9 : 0);
        const double v = so3_exp_jl_entry(wdt, lane < 9, e / 3, e % 3), vt = v * dt;
        if (lane < 18) E[lane] = sel64(lane < 9, v, vt);
    }
    __syncthreads();
    // T1 = F C: rows 3..5 (rotation: Rw and Jd entries) on threads 0..35, rows
    // 0..2 (C_i + dt C_{i+6}) on warp 2, rows 6..11 (C itself) on threads 128..199;
    // the noise terms on warp 3, the prior's quaternion on warp 7
    auto f_row = [&](const double* c, int stride, int a) {   // row 3 + a of F against a vector of C
        const double* r = E + 3 * a;
        const double* j = E + 9 + 3 * a;
        double s = r[0] * c[3 * stride];
        s = fma(r[1], c[4 * stride], s);
        s = fma(r[2], c[5 * stride], s);
        s = fma(j[0], c[9 * stride], s);
        s = fma(j[1], c[10 * stride], s);
        return fma(j[2], c[11 * stride], s);
    };
    if (tid < 36) {
        const double s = f_row(Cv + tid % 12, 12, tid / 12);
        T1[36 + tid] = s;
        bad = bad || !isfinite(s);
    } else if (warp == 2) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int e = lane + 32 * r;
            const double s = fma(dt, Cv[72 + (e < 36 ? e : 0)], Cv[e < 36 ? e : 0]);
            if (e < 36) {
                T1[e] = s;
                bad = bad || !isfinite(s);
            }
        }
    } else if (warp == 3) {
        // lanes 0..8: (Jd Qv Jd^T + Qp)_ab; 9: dt qv dt + qp; 10..18: Jd qv; 19: dt qv
        const int e = lane < 9 ? lane : 0, a = e / 3, b = e % 3;
        const double* ja = E + 9 + 3 * a;
        const double* jb = E + 9 + 3 * b;
        const bool pos = lane == 9, cross = lane >= 10 && lane < 19;
        const double q = qv[pos || lane == 19 ? 0 : 1];
        const double x0 = sel64(pos || lane == 19, dt, *(cross ? E + (lane - 1) : ja)) * q;
        const double x1 = ja[1] * q, x2 = ja[2] * q;
        const double s0 = x0 * sel64(pos, dt, jb[0]);
        const double s2 = fma(x2, jb[2], fma(x1, jb[1], s0));
        const double sp = P.sigma_pose[pos ? 0 : 1], qp = sp * sp;
        const double d = sel64(pos, s0, s2), dq = d + qp;
        if (lane < 10) nz[lane] = sel64(pos || a == b, dq, d);
        else if (lane < 20) nz[lane] = x0;
    } else if (tid >= 128 && tid < 200) {
        T1[72 + tid - 128] = Cv[72 + tid - 128];
    } else if (warp == 7) {   // the prior quaternion: normalise(quat_exp(wdt) (x) qm), component lane & 3
        const double qn = warp_quat_exp_mul(wd, qm);
        if (lane < 4) {
            dev->pq[lane] = qn;
            pose[3 + lane] = qn;
        }
    }
    bad = __syncthreads_or(bad) != 0;
    // F C F^T + noise, into Cv: column j of T1 F^T as T1 above
    if (tid < 36) {
        const int i = tid / 3, a = tid % 3;
        const double add = sel64(i >= 3 && i < 6, nz[i >= 3 && i < 6 ? 3 * (i - 3) + a : 0],
                                 sel64(i >= 9, nz[i >= 9 ? 10 + 3 * a + i - 9 : 0], 0.0));
        Cv[12 * i + 3 + a] = f_row(T1 + 12 * i, 1, a) + add;
    } else if (warp == 2) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
            const int e = lane + 32 * r, i = e < 36 ? e / 3 : 0, j = e % 3;
            const double add = sel64(i == j, nz[9], sel64(i == j + 6, nz[19], 0.0));
            const double s = fma(T1[12 * i + j + 6], dt, T1[12 * i + j]) + add;
            if (e < 36) Cv[12 * i + j] = s;
        }
    } else if (tid >= 128 && tid < 200) {
        const int i = (tid - 128) / 6, j = (tid - 128) % 6;
        const bool rot = i >= 3 && i < 6 && j >= 3;
        const double add = sel64(i < 3 && i == j, nz[19], sel64(rot, nz[rot ? 10 + 3 * (i - 3) + j - 3 : 0],
                                                                sel64(i == j + 6, qv[j < 3 ? 0 : 1], 0.0)));
        Cv[12 * i + 6 + j] = T1[12 * i + 6 + j] + add;
    } else if (warp == 7 && PREP != PREP_NONE) {
        warp_mats_rel(pose, anchor, dev->rel);
    } else if (warp == 3 && PREP != PREP_NONE) {
        // the localisation's constants: q0 = conj(q_anchor) (x) q_prior, b0 = Ra^T (t_prior - t_anchor)
        const int c = lane & 3, i2 = lane < 3 ? lane : 0;
        const double q0 = warp_quat_mul_component(sel64(c == 0, anchor[3], -anchor[3 + c]), pose + 3);
        const double b0 = fdot3(Ra[i2], pose[0] - anchor[0], Ra[3 + i2], pose[1] - anchor[1], Ra[6 + i2],
                                pose[2] - anchor[2]);
        if (lane < 4) dev->gn_q0[lane] = q0;
        if (lane < 3) dev->gn_b0[lane] = b0;
    }
    __syncthreads();
    if (tid < 78) {   // the symmetric part, one entry of the lower triangle a thread
        const int i = (int)((sqrtf(8.0f * (float)tid + 1.0f) - 1.0f) * 0.5f), j = tid - i * (i + 1) / 2;
        const double m = sel64(bad, __longlong_as_double(0x7ff8000000000000ll), 0.5 * (Cv[12 * i + j] + Cv[12 * j + i]));
        Sig[12 * i + j] = m;
        Sig[12 * j + i] = m;
        dev->pcov[12 * i + j] = m;
        dev->pcov[12 * j + i] = m;
        if (i < 6) {
            dev->cov_pp[6 * i + j] = m;
            dev->cov_pp[6 * j + i] = m;
        }
    } else if (PREP != PREP_NONE && warp == 3) {   // the start iterate's maps: J_l(0) = I
        if (lane < 9) {
            dev->gn_Ci[lane] = Ra[lane];
            dev->gn_Ci[9 + lane] = Ra[lane];
            dev->gn_Ji[lane] = lane % 4 == 0 ? 1.0 : 0.0;
        }
        if (lane < 6) dev->gn_m[lane] = 0.0;
    }
    __syncthreads();
    if (warp == 0) {   // the prior's precision
        int li = 0;
        if (lane < 21) {
#pragma unroll
            for (int i = 1; i < 6; ++i)
                if (lane >= tri6(i, 0)) li = i;
        }
        const int lm = lane < 21 ? lane - tri6(li, 0) : 0;
        bool pd;
        warp_spd6_inverse(Sig[12 * li + lm], &pd, Prec);
        if (lane == 0) ok = pd;
    }
    __syncthreads();
    if (!ok) {
        if (tid == 0) dev->flags |= FLAG_PRIOR_NOTPD;
        return;
    }
    const bool lp = PREP != PREP_NONE && tid >= 64 && tid < 128 && lane < 18;   // L' on warps 2 and 3, 18 entries each
    const int le = 18 * (warp & 1) + lane, pi = le / 6, pj = le % 6;
    if (tid < 36) {   // D = S_vp S_pp^-1
        const int i = tid / 6, j = tid % 6;
        double s = Sig[12 * (6 + i)] * Prec[j];
        for (int l = 1; l < 6; ++l) s = fma(Sig[12 * (6 + i) + l], Prec[6 * l + j], s);
        Dm[tid] = s;
        dev->D[tid] = s;
        dev->prec_pp[tid] = Prec[tid];
    } else if (lp) {  // L Ci, Ci = diag(Ra, Ra)
        const int b = pj / 3, jj = pj % 3;
        const double* L = Prec + 6 * pi + 3 * b;
        LC[le] = fdot3(L[0], Ra[jj], L[1], Ra[3 + jj], L[2], Ra[6 + jj]);
    }
    __syncthreads();
    if (tid < 36) {   // D S_pv
        const int i = tid / 6, j = tid % 6;
        double s = Dm[6 * i] * Sig[6 + j];
        for (int l = 1; l < 6; ++l) s = fma(Dm[6 * i + l], Sig[12 * l + 6 + j], s);
        W[tid] = s;
    } else if (lp) {  // L' = Ci^T (L Ci)
        const int b = pi / 3, ii = pi % 3;
        dev->gn_Lp[le] = fdot3(Ra[ii], LC[18 * b + pj], Ra[3 + ii], LC[18 * b + 6 + pj], Ra[6 + ii], LC[18 * b + 12 + pj]);
    }
    __syncthreads();
    if (tid < 36) {
        const int i = tid / 6, j = tid % 6;
        const double a = Sig[12 * (6 + i) + 6 + j] - W[tid], b = Sig[12 * (6 + j) + 6 + i] - W[6 * j + i];
        dev->cov_vel[tid] = 0.5 * (a + b);
    } else if (warp == 2) {
        if (lane < 6) dev->xi[lane] = 0.0;
        if (lane < 7) dev->cur_pose[lane] = pose[lane];
    }
}

// FP32 decision matrices of a pose (see PrepKind), computed once per pose by
// the FP64 recipe so that no kernel block repeats the FP64 chain; for
// PREP_REL also the Gauss-Newton tangent map of the current iterate (see
// track_dev.cuh), but for m (prep_vector_warp).  All 32 lanes of one warp call it;
// entries go one a lane.
__device__ __forceinline__ void prep_mats_warp(DevState* dev, int kind, const PoseArg& pose) {
    const int lane = threadIdx.x & 31;
    switch (kind) {
        case PREP_STATE:
            warp_mats_c2w(dev->t, dev->c2w);
            warp_mats_w2c(dev->t, dev->w2c);
            break;
        case PREP_AUX_C2W:
            warp_mats_c2w(pose.p, dev->aux);
            break;
        case PREP_AUX_REL:
            warp_mats_rel(pose.p, dev->anchor_pose, dev->aux);
            break;
        default: {
            const double* anchor = dev->anchor_pose;
            warp_mats_rel(dev->cur_pose, anchor, dev->rel);
            // Ra (lanes 0..8), then the prior's terms of the iterate in anchor-frame
            // coordinates
            const double* qa = anchor + 3;
            const double v = quat_R_entry_rn(qa[0], qa[1], qa[2], qa[3], lane < 9 ? lane : 0);
            __shared__ double s_ra[9], s_scr[63];
            if (lane < 9) {
                s_ra[lane] = v;
                dev->gn_Ci[lane] = v;
            }
            __syncwarp();
            warp_gn_prior_maps(s_ra, dev->prec_pp, dev->xi, dev->gn_Ci + 9, dev->gn_Lp, dev->gn_Ji, s_scr);
            // the localisation's constants: q0 = conj(q_anchor) (x) q_prior on
            // lanes 24..27, b0 = Ra^T (t_prior - t_anchor) on lanes 28..30
            const int c = lane & 3;
            const double q0 = warp_quat_mul_component(sel64(c == 0, qa[0], -qa[c]), dev->pq);
            if (lane >= 24 && lane < 28) dev->gn_q0[c] = q0;
            const int i2 = lane >= 28 && lane < 31 ? lane - 28 : 0;
            const double rb0 = __shfl_sync(0xffffffffu, v, i2), rb1 = __shfl_sync(0xffffffffu, v, 3 + i2),
                         rb2 = __shfl_sync(0xffffffffu, v, 6 + i2);
            const double b0 = fdot3(rb0, dev->pt[0] - anchor[0], rb1, dev->pt[1] - anchor[1], rb2,
                                    dev->pt[2] - anchor[2]);
            if (lane >= 28 && lane < 31) dev->gn_b0[i2] = b0;
        }
    }
}

// PREP_REL's m = Ci^T L xi, on a warp beside prep_mats_warp's.
__device__ __forceinline__ void prep_vector_warp(DevState* dev) {
    const int lane = threadIdx.x & 31;
    __shared__ double s_ra[9], s_scr[24];
    const double* qa = dev->anchor_pose + 3;
    const double v = quat_R_entry_rn(qa[0], qa[1], qa[2], qa[3], lane < 9 ? lane : 0);
    if (lane < 9) s_ra[lane] = v;
    __syncwarp();
    warp_gn_prior_vector(s_ra, dev->prec_pp, dev->xi, dev->gn_m, s_scr);
}

}  // namespace prism
