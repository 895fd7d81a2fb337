// Generalized surface regularization (GSR) at sample points, Eq. 9-13 (Sec. 3.3):
// the density of the 16 nearest splats (Eq. 9), the ideal flat density of the
// dominant splat g* (Eq. 10), the SDFs of both (Eq. 11), L_sdf (Eq. 12) and L_nor
// (Eq. 13), forward and analytic backward.
//
// k_gsr_prep turns each splat into an 80-byte record (centre, opacity, rotation,
// 1/s'^2, beta, smallest scale and its axis index), so a sample evaluates a
// neighbour from one record: the Mahalanobis form is taken in the splat's own axes,
// Q = sum_k (r_k . delta)^2 / s'_k^2, with no cancellation for flat splats (whose
// inverse covariance spans 1e4 to 1e8 in float32). k_gsr_sample runs one thread per
// sample: the sample's offset o = R_j (s'_j * z) from its splat's centre, the
// neighbour sums d and w (the direction of -grad d, relative to its largest term),
// g*, the losses, and then (a second pass over the neighbours, recomputing the
// per-neighbour terms instead of holding 16 sets in registers) the gradient with
// respect to each neighbour's centre, opacity, rotation, scales and beta, g*'s
// centre, axis, smallest scale and beta, and splat j's centre, rotation and scales
// (through x), all added into a 20-float accumulator per splat in the splats' own
// frames: the scale gradient of a flat axis is formed from that axis' projections,
// never recovered from a world-frame matrix gradient, where it would be a 1e-4 part
// cancelled out of the in-plane terms. k_gsr_chain takes each accumulator through
// s' = phi(beta) exp(l) and R(q) to the log-scales, beta and quaternion.
#include <cstring>

#include "ges_internal.cuh"
#include "splat_rec.cuh"

namespace ges {
namespace {

constexpr int kK = GES_KNN_K;
// Floats per splat accumulator: dL/d mu (3), o | R (9, row-major), s' (3) | beta, and three that stay 0, so that
// every accumulator is five aligned float4 and a neighbour's 17 values take five vector reductions.
constexpr int kAcc = 20;
constexpr int kGsrThreads = 128;
constexpr float kDMin = 1e-30f;
constexpr float kLn2 = 0.69314718055994531f;
constexpr float kHalfLog2e = 0.72134752044448170f;  // exp(-x/2) = exp2(-kHalfLog2e x)

struct GsrArgs {
    int n, m;
    int phi_mode;
    float rho;
    const float4 *pos_op, *lsb, *quat;
    const int32_t *knn;
    const int32_t *sample_splat;
    const float *sample_z;
    float lambda_sdf, lambda_nor, inv_m;
    float4 *rec;        // [n][kRec]
    float *acc;         // [n][kAcc], NULL: forward only
    double *partial;    // [blocks][2]
    float *losses;      // [3]
    float *sample_out;  // [m][8] or NULL
    float4 *g_pos_op, *g_lsb, *g_quat;
};

__device__ __forceinline__ void splat_frame(const GsrArgs &a, int i, float *R, float *sp, float &dphi, float &phi,
                                            float *es, float &qinv, float *qn) {
    ges::splat_frame(a.quat, a.lsb, a.rho, a.phi_mode, i, R, sp, dphi, phi, es, qinv, qn);
}

__global__ void __launch_bounds__(256) k_gsr_prep(GsrArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    build_splat_rec(a.pos_op, a.quat, a.lsb, a.rho, a.phi_mode, i, a.rec);
}

// Per-neighbour terms: delta = x - mu, v = A delta, Q = delta.v (as a sum over the
// axes), P = Q^(beta/2), G = exp(-P/2), t = o G. The weight of v in -grad d is
// t (beta/2) P / Q; relative to the largest term it is o exp(-(P - P_min)/2) (beta/2) P / Q.
struct NbTerms {
    float dx, dy, dz, vx, vy, vz, Q, lq, hb, P, G, t, o;
};

// (ox, oy, oz) is the sample's offset from the centre (cx, cy, cz) of the splat it was
// drawn from: delta = (centre - mu) + offset, so the sample's own splat sees its offset
// exactly and near neighbours a difference of nearby centres, which float32 represents
// without the cancellation of (centre + offset) - mu.
__device__ __forceinline__ NbTerms nb_terms(const NbRec &N, float cx, float cy, float cz, float ox, float oy,
                                           float oz) {
    NbTerms T;
    T.dx = (cx - N.r0.x) + ox; T.dy = (cy - N.r0.y) + oy; T.dz = (cz - N.r0.z) + oz;
    T.vx = T.vy = T.vz = 0.f;
    float Q = 0.f;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float p = N.R[k] * T.dx + N.R[3 + k] * T.dy + N.R[6 + k] * T.dz;
        const float ap = p * N.ia[k];
        Q = fmaf(ap, p, Q);
        T.vx = fmaf(ap, N.R[k], T.vx);
        T.vy = fmaf(ap, N.R[3 + k], T.vy);
        T.vz = fmaf(ap, N.R[6 + k], T.vz);
    }
    T.Q = Q;
    T.hb = 0.5f * N.beta;
    T.lq = log2f(T.Q);  // -inf at Q = 0
    T.P = exp2f(T.hb * T.lq);
    T.G = exp2f(-kHalfLog2e * T.P);
    T.o = N.r0.w;
    T.t = T.o * T.G;
    return T;
}

__device__ __forceinline__ void red_add(float *p, float v) {
    if (v != 0.f) atomicAdd(p, v);
}
// Adds four floats at a 16-byte aligned address with one reduction (each float on its own is atomic).
__device__ __forceinline__ void red_add4(float *p, float x, float y, float z, float w) {
    if (x != 0.f || y != 0.f || z != 0.f || w != 0.f)
        asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w)
                     : "memory");
}

// A warp's neighbour records in flight. A lane reading its own neighbour's 80 bytes touches a line of its own with
// each of five loads, and those lookups bound the kernel (L1 84 % busy); so the warp copies the 32 records
// of one neighbour slot together, consecutive lanes taking consecutive 16-byte pieces, two slots ahead,
// past L1 (a splat's neighbours are scattered: through L1 the copies of 20 warps evict one another, 1.76 ms).
// Forward and backward at 1.5M samples, the whole call: 1.41 ms with scalar reductions and own loads,
// 1.20 with vector reductions, 0.94 with staged records (two stages: 0.98; 7 CTAs per SM: 1.06), 0.90 with the
// accumulators cleared by a memory set and the sums added by 1,024 threads.
constexpr int kStages = 3;
struct GsrStage {
    int nb[32][GES_KNN_K + 1];       // the lanes' neighbour lists (padded: a column's entries in distinct banks)
    float4 rec[kStages][32][kRec];
};

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

// Starts copying the records of neighbour slot s (nothing past the last slot).
__device__ __forceinline__ void fetch_slot(GsrStage &S, const float4 *rec, int n, int s, int lane) {
    if (s < kK) {
        float4 *dst = &S.rec[s % kStages][0][0];
#pragma unroll
        for (int q = 0; q < kRec; ++q) {
            const int t = q * 32 + lane, r = t / kRec;
            const int i = S.nb[r][s];
            if (i >= 0 && i < n) cp_async16(dst + t, rec + kRec * (size_t)i + (t - kRec * r));
        }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}

// Waits for slot s (fetch_slot was called for the slots up to s + kStages - 2, each lane for its pieces).
__device__ __forceinline__ void await_slot() {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncwarp();
}

// Calls each(slot, neighbour's index, its record) for the lane's valid neighbours, in slot order.
template <class Each>
__device__ __forceinline__ void for_neighbours(GsrStage &S, const GsrArgs &a, int lane, Each &&each) {
#pragma unroll
    for (int s = 0; s < kStages - 1; ++s) fetch_slot(S, a.rec, a.n, s, lane);
    for (int s = 0; s < kK; ++s) {
        await_slot();
        // the slot fetched now lands where slot s - 1 was: every lane is past it (the wait above)
        fetch_slot(S, a.rec, a.n, s + kStages - 1, lane);
        const int i = S.nb[lane][s];
        if (i >= 0 && i < a.n) each(s, i, unpack_rec(S.rec[s % kStages][lane]));
    }
    __syncwarp();
}

__global__ void __launch_bounds__(kGsrThreads) k_gsr_sample(GsrArgs a) {
    __shared__ GsrStage s_stage[kGsrThreads / 32];
    const int k = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    GsrStage &S = s_stage[threadIdx.x >> 5];
    float l_sdf = 0.f, l_nor = 0.f;
    int j = k < a.m ? a.sample_splat[k] : -1;
    if (j >= a.n) j = -1;
    // the lists: 16 lanes to a list (a lane without a sample has an empty one)
#pragma unroll 4
    for (int r = 0; r < 32; r += 2) {
        const int jr = __shfl_sync(0xffffffffu, j, r + (lane >> 4));
        S.nb[r + (lane >> 4)][lane & 15] = jr >= 0 ? __ldg(a.knn + (size_t)jr * kK + (lane & 15)) : -1;
    }
    __syncwarp();
    float R[9], sp[3], es[3], qn[4], dphi, phi, qinv;
    const int jj = max(j, 0);
    splat_frame(a, jj, R, sp, dphi, phi, es, qinv, qn);
    const size_t kk = j >= 0 ? (size_t)k : 0;
    const float z0 = a.sample_z[3 * kk], z1 = a.sample_z[3 * kk + 1], z2 = a.sample_z[3 * kk + 2];
    const float4 pj = __ldg(a.pos_op + jj);
    const float m0 = sp[0] * z0, m1 = sp[1] * z1, m2 = sp[2] * z2;
    const float ox = R[0] * m0 + R[1] * m1 + R[2] * m2;  // x - mu_j
    const float oy = R[3] * m0 + R[4] * m1 + R[5] * m2;
    const float oz = R[6] * m0 + R[7] * m1 + R[8] * m2;
    // forward: d, g* (the smallest exponent P, first on ties: the largest falloff
    // exp(-P/2), decided where the falloffs themselves underflow), and -grad d's
    // direction w as a sum relative to the largest term exp(-P_min/2), rescaled
    // whenever a smaller P appears
    float d = 0.f, wx = 0.f, wy = 0.f, wz = 0.f, pmin = __int_as_float(0x7f800000);
    int best = -1;
    for_neighbours(S, a, lane, [&](int s, int, const NbRec &N) {
        const NbTerms T = nb_terms(N, pj.x, pj.y, pj.z, ox, oy, oz);
        d += T.t;
        if (T.P < pmin) {
            if (best >= 0) {
                const float sc = exp2f(-kHalfLog2e * (pmin - T.P));
                wx *= sc; wy *= sc; wz *= sc;
            }
            pmin = T.P;
            best = s;
        }
        const float ct = T.Q > 0.f ? T.o * exp2f(-kHalfLog2e * (T.P - pmin)) * T.hb * T.P / T.Q : 0.f;
        wx = fmaf(ct, T.vx, wx); wy = fmaf(ct, T.vy, wy); wz = fmaf(ct, T.vz, wz);
    });
    // what the backward walk needs of the losses' gradient
    float gd = 0.f, gwx = 0.f, gwy = 0.f, gwz = 0.f, gxx = 0.f, gxy = 0.f, gxz = 0.f;
    float gsx = 0.f, gsy = 0.f, gsz = 0.f, gn0 = 0.f, gn1 = 0.f, gn2 = 0.f, gsmin = 0.f, gbs = 0.f;
    int km = 0;
    if (best >= 0) {
        const int gs = S.nb[lane][best];
        const NbRec B = load_rec(a.rec, gs);
        const float n0 = B.km == 0 ? B.R[0] : (B.km == 1 ? B.R[1] : B.R[2]);
        const float n1 = B.km == 0 ? B.R[3] : (B.km == 1 ? B.R[4] : B.R[5]);
        const float n2 = B.km == 0 ? B.R[6] : (B.km == 1 ? B.R[7] : B.R[8]);
        const float ex = (pj.x - B.r0.x) + ox, ey = (pj.y - B.r0.y) + oy, ez = (pj.z - B.r0.z) + oz;
        const float e_raw = ex * n0 + ey * n1 + ez * n2;
        const float sg = e_raw < 0.f ? -1.f : 1.f;
        const float e = sg * e_raw;
        const float nsx = sg * n0, nsy = sg * n1, nsz = sg * n2;
        const float smin = B.smin, hs = 0.5f * B.beta;
        const float fbar = e > 0.f ? smin * exp2f(hs * log2f(e / smin)) : 0.f;
        const float dc = fminf(fmaxf(d, kDMin), 1.f);
        const float pl = -2.f * logf(dc);
        const float f = pl > 0.f ? smin * sqrtf(pl) : 0.f;
        const float wn = sqrtf(wx * wx + wy * wy + wz * wz);
        const float iw = wn > 0.f ? 1.f / wn : 0.f;
        const float ux = wx * iw, uy = wy * iw, uz = wz * iw;
        const float qx = ux - nsx, qy = uy - nsy, qz = uz - nsz;
        l_sdf = fabsf(fbar - f);
        l_nor = qx * qx + qy * qy + qz * qz;
        if (a.sample_out) {
            float *o = a.sample_out + 8 * (size_t)k;
            o[0] = pj.x + ox; o[1] = pj.y + oy; o[2] = pj.z + oz; o[3] = d; o[4] = f; o[5] = fbar;
            o[6] = ux * nsx + uy * nsy + uz * nsz;
            o[7] = (float)best;
        }
        if (a.acc) {
            const float gL = a.inv_m;
            const float gfb = a.lambda_sdf * gL * (fbar > f ? 1.f : (fbar < f ? -1.f : 0.f));
            const float gf = -gfb;
            // L_nor = |u - n*|^2
            const float gux = 2.f * a.lambda_nor * gL * qx, guy = 2.f * a.lambda_nor * gL * qy,
                        guz = 2.f * a.lambda_nor * gL * qz;
            const float gnsx = -gux, gnsy = -guy, gnsz = -guz;
            const float gud = gux * ux + guy * uy + guz * uz;
            gwx = (gux - gud * ux) * iw; gwy = (guy - gud * uy) * iw; gwz = (guz - gud * uz) * iw;
            // fbar = s_min^(1 - hs) e^hs
            float ge = 0.f;
            if (e > 0.f && smin > 0.f) {
                ge = gfb * hs * fbar / e;
                gsmin = gfb * (1.f - hs) * fbar / smin;
                gbs = 0.5f * gfb * fbar * logf(e / smin);
            }
            // f = s_min sqrt(-2 ln d)
            if (pl > 0.f && d > kDMin) {
                gsmin += gf * f / smin;
                gd = -gf * smin / (d * sqrtf(pl));
            }
            // e = sg (x - mu*) . n_raw, n* = sg n_raw; n_raw is column km of R*,
            // s_min is s'*[km]
            gxx = ge * nsx; gxy = ge * nsy; gxz = ge * nsz;
            gsx = gxx; gsy = gxy; gsz = gxz;
            km = B.km;
            // g*'s own terms join those it has as a neighbour (slot `best`)
            gn0 = sg * (ge * ex + gnsx);
            gn1 = sg * (ge * ey + gnsy);
            gn2 = sg * (ge * ez + gnsz);
        }
    }
    if (a.acc) {
        // neighbours: d = sum t_i (unscaled), w = sum ct_i v_i (relative weights)
        for_neighbours(S, a, lane, [&](int s, int i, const NbRec &N) {
            if (best < 0) return;
            const NbTerms T = nb_terms(N, pj.x, pj.y, pj.z, ox, oy, oz);
            const float iq = T.Q > 0.f ? 1.f / T.Q : 0.f;
            const float er = exp2f(-kHalfLog2e * (T.P - pmin));
            const float ct = T.o * er * T.hb * T.P * iq;  // relative weight of v in w
            const float gc = gwx * T.vx + gwy * T.vy + gwz * T.vz;
            const float gvx = ct * gwx, gvy = ct * gwy, gvz = ct * gwz;
            const float lnq = T.Q > 0.f ? T.lq * kLn2 : 0.f;
            // the density path (t = o G) and the direction path (ct)
            const float go = gd * T.G + gc * er * T.hb * T.P * iq;
            const float gQ = -0.5f * gd * T.t * T.hb * T.P * iq +
                             gc * ct * ((T.hb - 1.f) * iq - 0.5f * T.hb * T.P * iq);
            const float ghb = -0.5f * gd * T.t * T.P * lnq +
                              gc * ct * ((T.hb > 0.f ? 1.f / T.hb : 0.f) + lnq - 0.5f * T.P * lnq);
            // Q = sum_k a_k p_k^2 and v = sum_k a_k p_k r_k with p_k = r_k . delta,
            // a_k = 1/s'_k^2: per axis h_k = 2 gQ a_k p_k + a_k (r_k . g_v);
            // dL/ddelta = sum_k h_k r_k, dL/dr_k = h_k delta + a_k p_k g_v,
            // dL/da_k = gQ p_k^2 + p_k (r_k . g_v)
            float gdx = 0.f, gdy = 0.f, gdz = 0.f, GR[9], gsp[3];
            const bool star = s == best;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float r0c = N.R[c], r1c = N.R[3 + c], r2c = N.R[6 + c], ak = N.ia[c];
                const float pk = r0c * T.dx + r1c * T.dy + r2c * T.dz;
                const float gk = r0c * gvx + r1c * gvy + r2c * gvz;
                const float hk = 2.f * gQ * ak * pk + ak * gk;
                gdx = fmaf(hk, r0c, gdx); gdy = fmaf(hk, r1c, gdy); gdz = fmaf(hk, r2c, gdz);
                const float apk = ak * pk;
                const bool axis = star && km == c;
                GR[c] = hk * T.dx + apk * gvx + (axis ? gn0 : 0.f);
                GR[3 + c] = hk * T.dy + apk * gvy + (axis ? gn1 : 0.f);
                GR[6 + c] = hk * T.dz + apk * gvz + (axis ? gn2 : 0.f);
                const float gak = gQ * pk * pk + pk * gk;
                gsp[c] = gak * (-2.f * ak * sqrtf(ak)) + (axis ? gsmin : 0.f);  // da/ds' = -2 / s'^3
            }
            gxx += gdx; gxy += gdy; gxz += gdz;
            float *ai = a.acc + (size_t)i * kAcc;
            red_add4(ai, star ? -gdx - gsx : -gdx, star ? -gdy - gsy : -gdy,
                     star ? -gdz - gsz : -gdz, go);
            red_add4(ai + 4, GR[0], GR[1], GR[2], GR[3]);
            red_add4(ai + 8, GR[4], GR[5], GR[6], GR[7]);
            red_add4(ai + 12, GR[8], gsp[0], gsp[1], gsp[2]);
            red_add(ai + 16, 0.5f * ghb + (star ? gbs : 0.f));
        });
        if (best >= 0) {  // x = mu_j + R diag(s') z
            float *aj = a.acc + (size_t)j * kAcc;
            const float gxv[3] = {gxx, gxy, gxz}, zv[3] = {z0, z1, z2};
            float GR[9], gsp[3];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
#pragma unroll
                for (int r = 0; r < 3; ++r) GR[3 * r + c] = gxv[r] * zv[c] * sp[c];
                gsp[c] = zv[c] * (R[c] * gxx + R[3 + c] * gxy + R[6 + c] * gxz);
            }
            red_add4(aj, gxx, gxy, gxz, 0.f);
            red_add4(aj + 4, GR[0], GR[1], GR[2], GR[3]);
            red_add4(aj + 8, GR[4], GR[5], GR[6], GR[7]);
            red_add4(aj + 12, GR[8], gsp[0], gsp[1], gsp[2]);
        }
    }
    // CTA sums of the two loss terms (double), in a fixed order
    __shared__ double s_red[2][kGsrThreads / 32];
    double d0 = l_sdf, d1 = l_nor;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        d0 += __shfl_down_sync(0xffffffffu, d0, o);
        d1 += __shfl_down_sync(0xffffffffu, d1, o);
    }
    if ((threadIdx.x & 31) == 0) { s_red[0][threadIdx.x >> 5] = d0; s_red[1][threadIdx.x >> 5] = d1; }
    __syncthreads();
    if (threadIdx.x == 0) {
        double t0 = 0.0, t1 = 0.0;
        for (int w = 0; w < kGsrThreads / 32; ++w) { t0 += s_red[0][w]; t1 += s_red[1][w]; }
        a.partial[2 * (size_t)blockIdx.x] = t0;
        a.partial[2 * (size_t)blockIdx.x + 1] = t1;
    }
}

// One CTA adds the CTAs' partial sums in a fixed order (its length is the loads' latency: 1,024 threads take a
// quarter of the rounds of 256).
__global__ void __launch_bounds__(1024) k_gsr_finalize(GsrArgs a, int nblocks) {
    __shared__ double s0[1024], s1[1024];
    const int t = threadIdx.x;
    double x0 = 0.0, x1 = 0.0;
    for (int b = t; b < nblocks; b += 1024) {
        const double2 p = reinterpret_cast<const double2 *>(a.partial)[b];
        x0 += p.x;
        x1 += p.y;
    }
    s0[t] = x0;
    s1[t] = x1;
    __syncthreads();
    for (int o = 512; o > 0; o >>= 1) {
        if (t < o) { s0[t] += s0[t + o]; s1[t] += s1[t + o]; }
        __syncthreads();
    }
    if (t == 0) {
        const double m = (double)a.m;
        a.losses[0] = (float)(s0[0] / m);
        a.losses[1] = (float)(s1[0] / m);
        a.losses[2] = (float)((double)a.lambda_sdf * s0[0] / m + (double)a.lambda_nor * s1[0] / m);
    }
}

// Accumulated gradients of (mu, o, R, s', beta) -> (pos_op, lscale_beta, quat).
__global__ void __launch_bounds__(256) k_gsr_chain(GsrArgs a) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.n) return;
    float R[9], sp[3], es[3], qn[4], dphi, phi, qinv;
    splat_frame(a, i, R, sp, dphi, phi, es, qinv, qn);
    const float4 *g4 = reinterpret_cast<const float4 *>(a.acc + (size_t)i * kAcc);
    const float4 a0 = g4[1], a1 = g4[2], a2 = g4[3];
    a.g_pos_op[i] = g4[0];
    const float GR[9] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w, a2.x}, gs3[3] = {a2.y, a2.z, a2.w};
    // s' = phi(beta) exp(l)
    float gbeta = a.acc[(size_t)i * kAcc + 16];
    float gl[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        gl[c] = gs3[c] * sp[c];
        gbeta += gs3[c] * dphi * es[c];
    }
    a.g_lsb[i] = make_float4(gl[0], gl[1], gl[2], gbeta);
    // R(q) -> unit quaternion -> quaternion
    const float w = qn[0], x = qn[1], y = qn[2], z = qn[3];
    const float gw = 2.f * (-z * GR[1] + y * GR[2] + z * GR[3] - x * GR[5] - y * GR[6] + x * GR[7]);
    const float gx = 2.f * (y * GR[1] + z * GR[2] + y * GR[3] - 2.f * x * GR[4] - w * GR[5] + z * GR[6] + w * GR[7] -
                            2.f * x * GR[8]);
    const float gy = 2.f * (-2.f * y * GR[0] + x * GR[1] + w * GR[2] + x * GR[3] + z * GR[5] - w * GR[6] + z * GR[7] -
                            2.f * y * GR[8]);
    const float gz = 2.f * (-2.f * z * GR[0] - w * GR[1] + x * GR[2] + w * GR[3] - 2.f * z * GR[4] + y * GR[5] +
                            x * GR[6] + y * GR[7]);
    const float dq = gw * w + gx * x + gy * y + gz * z;
    a.g_quat[i] = make_float4((gw - w * dq) * qinv, (gx - x * dq) * qinv, (gy - y * dq) * qinv, (gz - z * dq) * qinv);
}

struct GsrLayout {
    uint64_t rec, acc, partial, bytes;
    uint32_t nblocks;
};

inline uint64_t al256g(uint64_t x) { return (x + 255) & ~uint64_t(255); }

GsrLayout gsr_layout(int32_t n, int32_t m) {
    GsrLayout L;
    L.nblocks = ceil_div_u64(m > 0 ? (uint64_t)m : 1, kGsrThreads);
    uint64_t off = 0;
    L.rec = off; off = al256g(off + 16ull * kRec * n);
    L.acc = off; off = al256g(off + 4ull * kAcc * n);
    L.partial = off; off = al256g(off + 16ull * L.nblocks);
    L.bytes = off;
    return L;
}

}  // namespace
}  // namespace ges

using namespace ges;

extern "C" size_t ges_gsr_workspace_bytes(int32_t n, int32_t m) {
    if (n < 1 || m < 1 || (uint64_t)n > (1ull << 26) || (uint64_t)m > (1ull << 28)) return 0;
    return gsr_layout(n, m).bytes;
}

extern "C" ges_status ges_gsr(int32_t n, const float *pos_op, const float *lscale_beta, const float *quat,
                              const ges_config *cfg, const int32_t *knn, int32_t m, const int32_t *sample_splat,
                              const float *sample_z, float lambda_sdf, float lambda_nor, void *workspace,
                              size_t workspace_bytes, float *losses, float *sample_out, float *g_pos_op,
                              float *g_lscale_beta, float *g_quat, void *stream) {
    GES_RANGE();
    if (n < 1 || m < 1 || (uint64_t)n > (1ull << 26) || (uint64_t)m > (1ull << 28)) return GES_ERR_INVALID_ARG;
    if (!pos_op || !lscale_beta || !quat || !cfg || !knn || !sample_splat || !sample_z || !workspace || !losses)
        return GES_ERR_INVALID_ARG;
    const bool grads = g_pos_op || g_lscale_beta || g_quat;
    if (grads && !(g_pos_op && g_lscale_beta && g_quat)) return GES_ERR_INVALID_ARG;
    for (const void *p : {(const void *)pos_op, (const void *)lscale_beta, (const void *)quat, (const void *)g_pos_op,
                          (const void *)g_lscale_beta, (const void *)g_quat})
        if ((uintptr_t)p & 15u) return GES_ERR_INVALID_ARG;
    if (((uintptr_t)workspace & 255u) || cfg->phi_mode < 0 || cfg->phi_mode > 2 || !isfinite(cfg->rho))
        return GES_ERR_INVALID_ARG;
    if (!isfinite(lambda_sdf) || !isfinite(lambda_nor)) return GES_ERR_INVALID_ARG;
    const GsrLayout L = gsr_layout(n, m);
    if (workspace_bytes < L.bytes) return GES_ERR_INVALID_ARG;
    GsrArgs a;
    memset(&a, 0, sizeof(a));
    a.n = n; a.m = m; a.phi_mode = cfg->phi_mode; a.rho = cfg->rho;
    a.pos_op = reinterpret_cast<const float4 *>(pos_op);
    a.lsb = reinterpret_cast<const float4 *>(lscale_beta);
    a.quat = reinterpret_cast<const float4 *>(quat);
    a.knn = knn; a.sample_splat = sample_splat; a.sample_z = sample_z;
    a.lambda_sdf = lambda_sdf; a.lambda_nor = lambda_nor; a.inv_m = (float)(1.0 / (double)m);
    char *ws = static_cast<char *>(workspace);
    a.rec = reinterpret_cast<float4 *>(ws + L.rec);
    a.acc = grads ? reinterpret_cast<float *>(ws + L.acc) : nullptr;
    a.partial = reinterpret_cast<double *>(ws + L.partial);
    a.losses = losses; a.sample_out = sample_out;
    a.g_pos_op = reinterpret_cast<float4 *>(g_pos_op);
    a.g_lsb = reinterpret_cast<float4 *>(g_lscale_beta);
    a.g_quat = reinterpret_cast<float4 *>(g_quat);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (grads && cudaMemsetAsync(a.acc, 0, 4ull * kAcc * (uint64_t)n, s) != cudaSuccess) return GES_ERR_CUDA;
    k_gsr_prep<<<ceil_div_u64(n, 256), 256, 0, s>>>(a);
    k_gsr_sample<<<L.nblocks, kGsrThreads, 0, s>>>(a);
    k_gsr_finalize<<<1, 1024, 0, s>>>(a, (int)L.nblocks);
    if (grads) k_gsr_chain<<<ceil_div_u64(n, 256), 256, 0, s>>>(a);
    return cudaGetLastError() == cudaSuccess ? GES_OK : GES_ERR_CUDA;
}
