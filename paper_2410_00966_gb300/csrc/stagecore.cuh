// Device code shared by the stage kernels (stage.cu, xinv.cu): Runge-Kutta
// tableaux, the per-cell field / torque / RK update, the block
// reductions and the per-instance FP64 scalar work.  Included by each translation
// unit; constant-memory tables are per unit and filled by upload_tableaux().
#pragma once

#include <math.h>

#include "common.cuh"
#include "kern_common.cuh"

namespace mq {

// Butcher tableaux: [kind][stage][j].
static __constant__ float c_af[2][MAX_STAGES][MAX_STAGES];
static __constant__ double c_ad[2][MAX_STAGES][MAX_STAGES];
static __constant__ float c_bf[2][MAX_STAGES];    // weights of the propagated solution
static __constant__ double c_bd[2][MAX_STAGES];
static __constant__ double c_cd[2][MAX_STAGES];   // stage times
static __constant__ float c_ef[MAX_STAGES];       // DP45 error weights b5 - b4

__device__ __forceinline__ double warp_sum_d(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}
__device__ __forceinline__ float warp_max_f(float v) {
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_down_sync(0xffffffffu, v, o));
    return v;
}
// Fixed-shape block reduction (deterministic for a given blockDim).
static __device__ double block_sum_d(double v, double* red) {
    v = warp_sum_d(v);
    int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    if (l == 0) red[w] = v;
    __syncthreads();
    int nw = (blockDim.x + 31) >> 5;
    double r = 0.0;
    if (w == 0) {
        r = l < nw ? red[l] : 0.0;
        r = warp_sum_d(r);
    }
    __syncthreads();
    return r;  // valid in thread 0
}

// A sum kept as three floats: the rounding error of each addition to h is
// computed exactly (Knuth's two-sum), that of the addition of those errors to m
// likewise, and what is left goes to l.  Wider than the 53 bits of an FP64
// accumulator, from FP32 additions only: this part issues two FP64 lanes per SM
// and clock, so that an FP64 add and conversion per cell took 32 of its clocks
// per warp against 3, and each of the ten dependent FP64 adds of a block
// reduction about 300 clocks of latency against 100.
// Every rounding is written out: a term that the compiler fuses as a product
// into one addition of the two-sum and not into the other leaves an error of
// 2^-24 of the term (3e-11 of the sum of |terms| over 60000 cells).
struct Sum3 {
    float h, m, l;
};
__device__ __forceinline__ float two_sum(float& a, float b) {   // a += b; the exact error
    const float t = __fadd_rn(a, b), z = __fsub_rn(t, a);
    const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(b, z));
    a = t;
    return e;
}
__device__ __forceinline__ void sum3_add(Sum3& s, float x) {
    const float e = two_sum(s.h, x);
    s.l = __fadd_rn(s.l, two_sum(s.m, e));
}
// s += x y, the product exact (its rounding error is the fused remainder).
__device__ __forceinline__ void sum3_add_product(Sum3& s, float x, float y) {
    const float p = __fmul_rn(x, y), q = __fmaf_rn(x, y, -p);
    const float e = two_sum(s.h, p), f = two_sum(s.m, e);
    s.l = __fadd_rn(s.l, __fadd_rn(f, two_sum(s.m, q)));
}
__device__ __forceinline__ void sum3_merge(Sum3& s, const Sum3& o) {
    const float e = two_sum(s.h, o.h), f = two_sum(s.m, o.m);
    s.l = __fadd_rn(__fadd_rn(s.l, o.l), __fadd_rn(f, two_sum(s.m, e)));
}
__device__ __forceinline__ double sum3_value(const Sum3& s) { return (double)s.h + ((double)s.m + (double)s.l); }
__device__ __forceinline__ Sum3 warp_sum3(Sum3 v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        Sum3 w;
        w.h = __shfl_down_sync(0xffffffffu, v.h, o);
        w.m = __shfl_down_sync(0xffffffffu, v.m, o);
        w.l = __shfl_down_sync(0xffffffffu, v.l, o);
        sum3_merge(v, w);
    }
    return v;
}
__device__ __forceinline__ float4 sum3_pack(const Sum3& s) { return make_float4(s.h, s.m, s.l, 0.f); }
__device__ __forceinline__ Sum3 sum3_unpack(const float4& f) { return Sum3{f.x, f.y, f.z}; }

// Sums of the NQ terms and the maximum of the float (with_max, uniform) of
// every thread, in one block barrier for all of them: the results are valid
// in thread 0.  `red` holds NQ rows and `redf` one row of 32 warp values; the
// caller synchronises before they are written again.  Fixed order for a given
// blockDim.
template <int NQ>
static __device__ __forceinline__ void block_reduce(Sum3 (&v)[NQ], float& mx, bool with_max, float4* red,
                                                    float* redf) {
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31, nw = (blockDim.x + 31) >> 5;
#pragma unroll
    for (int q = 0; q < NQ; q++) v[q] = warp_sum3(v[q]);
    if (with_max) mx = warp_max_f(mx);
    if (l == 0) {
#pragma unroll
        for (int q = 0; q < NQ; q++) red[q * 32 + w] = sum3_pack(v[q]);
        redf[w] = mx;
    }
    __syncthreads();
    if (w == 0) {
#pragma unroll
        for (int q = 0; q < NQ; q++) v[q] = warp_sum3(l < nw ? sum3_unpack(red[q * 32 + l]) : Sum3{0.f, 0.f, 0.f});
        if (with_max) mx = warp_max_f(l < nw ? redf[l] : 0.f);
    }
}

// Gamma_k from the P-mode accumulators, Eq. (gammadiscretefinal), with e =
// exp(-kappa t), sn and cs the sine and cosine of omega t.
static __device__ double gamma_p(const InstParams& ip, const InstState& s, int k, double e, double sn, double cs,
                                 double hbar) {
    return e * cs * (ip.x0[k] - 2.0 * s.S[k] / hbar) - e * sn * (ip.p0[k] - 2.0 * s.C[k] / hbar);
}

// FP64 scalar work of one instance at the end of stage k, by one warp: lane
// q < A.nmodes does mode q's arithmetic -- the amplitude (E-mode: d alpha_k/dt
// = -(kappa_k + i omega_k) alpha_k + i X_k / hbar, Eq. eqmotionaclasical with
// omega_c -> omega_c - i kappa) or the accumulators (P-mode, Eq. Sdiscrete /
// Cdiscrete) -- and lane 0 also time, accept / reject and step size.
// load(): everything that does not depend on this stage's coupling sums: the
// state (independent loads) and the Runge-Kutta sums over the earlier stages,
// to run while the partials are on their way.  finish(): the rest, as few
// dependent FP64 operations as it takes (about 300 clocks each).  (One thread that copied the 750-byte state to its
// stack and then did every mode took 4.7 us of a 20 us x inverse.)
struct StageFinish {
    double dt, tcav;
    double re, im;       // E-mode: alpha_q plus the terms of the stages before k
    double ar, ai;       // E-mode: alpha_q of stage k
    double dr, di;       // E-mode: its derivative without X / hbar
    double w;            // dt times the weight of stage k
    bool cav, amp, last;

    __device__ __forceinline__ void load(const StageArgs& A, int k, const InstParams& ip, const InstState& s) {
        const int q = threadIdx.x & 31, K = A.kind;
        cav = q < A.nmodes && ip.cav_on[q < MAX_MODES ? q : 0] != 0;
        amp = cav && A.mode == CAV_E;
        last = k == (K == KIND_RK4 ? 3 : 6);
        dt = s.dt;
        tcav = s.tcav;
        re = im = ar = ai = dr = di = w = 0.0;
        if (!amp) return;
        double kr[MAX_STAGES - 1], ki[MAX_STAGES - 1];
#pragma unroll
        for (int j = 0; j < MAX_STAGES - 1; j++) {
            kr[j] = j < k ? s.ka_re[q][j] : 0.0;
            ki[j] = j < k ? s.ka_im[q][j] : 0.0;
        }
        re = s.a_re[q];
        im = s.a_im[q];
        // stage 1 is at alpha itself (as_re holds the amplitude of the stage
        // after the last launched one, which a host-side change may follow)
        ar = (k == 0 ? s.a_re : s.as_re)[q];
        ai = (k == 0 ? s.a_im : s.as_im)[q];
        dr = -ip.kappa[q] * ar + ip.wc[q] * ai;
        di = -ip.kappa[q] * ai - ip.wc[q] * ar;
        // weights of the next stage (DP45 stage 7: the 5th-order ones), or of
        // the step (RK4's last stage; DP45's last is already its alpha5)
        if (last && K == KIND_DP45) return;
        const double* c = last || (K == KIND_DP45 && k == 5) ? c_bd[K] : c_ad[K][k + 1];
#pragma unroll
        for (int j = 0; j < MAX_STAGES - 1; j++)
            if (j < k) {
                re += dt * c[j] * kr[j];
                im += dt * c[j] * ki[j];
            }
        w = dt * c[k];
    }

    // Xsum: the mode's coupling sum without V_c (lane q); errmax uniform over
    // the warp; msum read by lane 0; trig[0..2][q] (P-mode, last stage):
    // exp(kappa t), sin and cos of omega t at the end of the step.
    __device__ __forceinline__ void finish(const Material& mat, const StageArgs& A, int k, const InstParams& ip,
                                           InstState& s, double Xsum, float errmax, double* hist, int hcap, int* flags,
                                           const double* msum, double* mhist, const double (*trig)[MAX_MODES]) {
        const int q = threadIdx.x & 31, K = A.kind;
        const double X = Xsum * mat.vc;
        if (q < A.nmodes) s.X[q] = X;
        if (amp) {
            di = fma(Xsum, mat.vc_hbar, di);
            s.ka_re[q][k] = dr;
            s.ka_im[q][k] = di;
            // (not at DP45's last stage: a rejected attempt may have overflowed,
            // and alpha_q must stay what it was)
            if (!(last && K == KIND_DP45)) {
                re += w * dr;
                im += w * di;
            }
        }
        if (!last) {
            if (amp) {
                s.as_re[q] = ar = re;
                s.as_im[q] = ai = im;
            }
            if (q == 0 && K == KIND_DP45 && k == 0) s.have_k1 = 1;
            return;
        }
        bool accept = true;
        double nd = dt;                     // next step length
        if (K == KIND_DP45) {
            if (s.poison || !(errmax == errmax)) errmax = INFINITY;
            accept = errmax <= A.tol;
            const double err = (double)errmax;
            double f = err > 0.0 ? 0.9 * pow((double)A.tol / err, 0.2) : 5.0;
            if (!(f == f)) f = 0.2;
            f = fmin(5.0, fmax(0.2, f));
            nd = dt * f;
            const double t = accept ? s.t + dt : s.t, te = s.t_end;
            bool done = false;
            if (te > 0.0) {
                if (t >= te * (1.0 - 1e-14)) done = true;
                else if (t + nd > te) nd = te - t;
            }
            if (nd < 1e-20 && !done) {
                if (q == 0) atomicOr(flags, FLAG_DT_UNDERFLOW);
                done = true;
            }
            __syncwarp();                   // every lane has read the state
            if (q == 0) {
                s.err = err;
                s.poison = 0;
                if (done) s.done = 1;
                s.dt = nd;
            }
        }
        if (amp) {
            if (K == KIND_DP45 && accept) {
                re = ar;                    // alpha5
                im = ai;
                s.ka_re[q][0] = dr;
                s.ka_im[q][0] = di;
            }
            if (accept) {
                s.a_re[q] = re;
                s.a_im[q] = im;
            }
            ar = re;                        // amplitude of the next step's stage 1
            ai = im;
        } else if (cav && accept) {
            s.S[q] += trig[0][q] * trig[1][q] * X * dt;
            s.C[q] += trig[0][q] * trig[2][q] * X * dt;
        }
        if (q == 0) {
            if (accept) {
                if (K == KIND_DP45) {
                    s.mcur ^= 1;
                    s.k1slot = s.k1slot == 0 ? 6 : 0;
                    if (A.mode == CAV_P) s.have_k1 = 0;   // Gamma at t_n changes with S_n, C_n
                }
                s.t += dt;
                s.tcav = tcav + dt;
                s.nacc++;
                if (s.nhist < hcap) hist[s.nhist] = dt;
                else atomicOr(flags, FLAG_HIST_FULL);
                s.nhist++;
                if (A.record > 0 && mhist && s.nacc % A.record == 0) {
                    if (s.nmh < hcap) {
                        double* e = mhist + 4 * s.nmh;
                        e[0] = s.t;
                        for (int c = 0; c < 3; c++) e[1 + c] = msum[c] * ip.inv_nmag;
                    } else {
                        atomicOr(flags, FLAG_HIST_FULL);
                    }
                    s.nmh++;
                }
            } else {
                s.nrej++;
            }
        }
    }
};

static void upload_tableaux() {
    float af[2][MAX_STAGES][MAX_STAGES] = {};
    double ad[2][MAX_STAGES][MAX_STAGES] = {};
    float bf[2][MAX_STAGES] = {};
    double bd[2][MAX_STAGES] = {};
    double cd[2][MAX_STAGES] = {};
    float ef[MAX_STAGES] = {};
    // classic RK4
    ad[0][1][0] = 0.5; ad[0][2][1] = 0.5; ad[0][3][2] = 1.0;
    double b4[4] = {1.0 / 6, 1.0 / 3, 1.0 / 3, 1.0 / 6};
    double c4[4] = {0.0, 0.5, 0.5, 1.0};
    for (int j = 0; j < 4; j++) { bd[0][j] = b4[j]; cd[0][j] = c4[j]; }
    // Dormand & Prince (1980) RK5(4)7FM
    const double A5[7][6] = {
        {0, 0, 0, 0, 0, 0},
        {1.0 / 5, 0, 0, 0, 0, 0},
        {3.0 / 40, 9.0 / 40, 0, 0, 0, 0},
        {44.0 / 45, -56.0 / 15, 32.0 / 9, 0, 0, 0},
        {19372.0 / 6561, -25360.0 / 2187, 64448.0 / 6561, -212.0 / 729, 0, 0},
        {9017.0 / 3168, -355.0 / 33, 46732.0 / 5247, 49.0 / 176, -5103.0 / 18656, 0},
        {35.0 / 384, 0, 500.0 / 1113, 125.0 / 192, -2187.0 / 6784, 11.0 / 84}};
    const double B5[7] = {35.0 / 384, 0, 500.0 / 1113, 125.0 / 192, -2187.0 / 6784, 11.0 / 84, 0};
    const double B4[7] = {5179.0 / 57600, 0, 7571.0 / 16695, 393.0 / 640, -92097.0 / 339200, 187.0 / 2100, 1.0 / 40};
    const double C5[7] = {0, 1.0 / 5, 3.0 / 10, 4.0 / 5, 8.0 / 9, 1, 1};
    for (int s = 0; s < 7; s++)
        for (int j = 0; j < 6; j++) ad[1][s][j] = A5[s][j];
    for (int j = 0; j < 7; j++) { bd[1][j] = B5[j]; cd[1][j] = C5[j]; ef[j] = (float)(B5[j] - B4[j]); }
    for (int k = 0; k < 2; k++) {
        for (int s = 0; s < 7; s++) for (int j = 0; j < 7; j++) af[k][s][j] = (float)ad[k][s][j];
        for (int j = 0; j < 7; j++) bf[k][j] = (float)bd[k][j];
    }
    cudaMemcpyToSymbol(c_af, af, sizeof(af));
    cudaMemcpyToSymbol(c_ad, ad, sizeof(ad));
    cudaMemcpyToSymbol(c_bf, bf, sizeof(bf));
    cudaMemcpyToSymbol(c_bd, bd, sizeof(bd));
    cudaMemcpyToSymbol(c_cd, cd, sizeof(cd));
    cudaMemcpyToSymbol(c_ef, ef, sizeof(ef));
}


// Stage input m_s = m0 + dt sum_j a_sj k_j of the Runge-Kutta stage being
// evaluated (Eq. llg integrated by RK4 / Dormand-Prince).  At the last
// Dormand-Prince stage the 5th-order solution is formed, renormalised and
// stored as the candidate, with the partial error dt sum_j e_j k_j.
// Weights are indexed by compile-time stage numbers only (registers, no
// stack), and the k buffers are read through the kernel's parameter block.
struct StageInput {
    float kw[MAX_STAGES - 1], ke[MAX_STAGES - 1];
    const float4* k0;    // buffer of stage 1 (DP45: first-same-as-last slot)
    long long base;
    bool form, dp_last;
    float4* out;         // where m_s is written (stage > 0)
    float4* e6;

    // apply() takes the cell index relative to `base` (the block's first cell).
    __device__ __forceinline__ void init(const Buffers& Bf, const StageArgs& A, const InstState& st, long long base_) {
        const int s = A.stage;
        const float dt = (float)st.dt;
        base = base_;
        form = !A.field_only && s > 0;
        dp_last = A.kind == KIND_DP45 && s == 6 && !A.field_only;
#pragma unroll
        for (int j = 0; j < MAX_STAGES - 1; j++) {
            const bool on = form && j < s;
            kw[j] = on ? dt * (dp_last ? c_bf[1][j] : c_af[A.kind][s][j]) : 0.f;
            ke[j] = on && dp_last ? dt * c_ef[j] : 0.f;
        }
        k0 = (A.kind == KIND_DP45 ? Bf.k[st.k1slot] : Bf.k[0]) + base;
        out = (dp_last ? Bf.m[st.mcur ^ 1] : Bf.ms) + base;
        e6 = Bf.e6 + base;
    }

    // Ask L2 for the k rows this block will read ([base, base + bytes) of each).
    __device__ __forceinline__ void prefetch(const Buffers& Bf, unsigned bytes) const {
        if (!form) return;
#pragma unroll
        for (int q = 0; q < MAX_STAGES - 1; q++)
            if (kw[q] != 0.f || ke[q] != 0.f) prefetch_l2(q == 0 ? k0 : Bf.k[q] + base, bytes);
    }

    // v = m0[i] on entry; m_s on return (written to out, and e6 at the last DP stage)
    __device__ __forceinline__ void apply(const Buffers& Bf, float4& v, int i) const {
        if (!form) return;
        float ax = 0.f, ay = 0.f, az = 0.f, ex = 0.f, ey = 0.f, ez = 0.f;
#pragma unroll
        for (int q = 0; q < MAX_STAGES - 1; q++) {
            if (kw[q] != 0.f || ke[q] != 0.f) {
                const float4 kj = q == 0 ? k0[i] : Bf.k[q][base + i];
                ax += kw[q] * kj.x; ay += kw[q] * kj.y; az += kw[q] * kj.z;
                ex += ke[q] * kj.x; ey += ke[q] * kj.y; ez += ke[q] * kj.z;
            }
        }
        v.x += ax; v.y += ay; v.z += az;
        if (dp_last) {
            float r2 = v.x * v.x + v.y * v.y + v.z * v.z;
            float inv = r2 > 0.f ? rsqrtf(r2) : 0.f;
            v.x *= inv; v.y *= inv; v.z *= inv;
            e6[i] = make_float4(ex, ey, ez, 0.f);
        }
        out[i] = v;
    }
};

// Everything a stage needs per cell once demag and exchange are known:
// anisotropy, Zeeman (with the Appendix C excitation) and cavity fields, the
// LLG torque (Eq. llg), the RK bookkeeping of this stage, and the cell's
// share of the coupling sums and of the DP45 error.  NM: cavity modes
// compiled in (1: the paper's single mode; MAX_MODES: up to A.nmodes).
// Material constants and buffer pointers are read from the kernel's
// parameter block at each use.
template <int NM>
struct CellUpdate {
    float G[NM], bs[NM];
    bool on[NM];
    float dt, bex, bey, bez, D;
    bool want_demag, want_exch, want_anis, want_zee, want_cav, field_only;
    int K, s, mode, nm;
    long long cb, fb;    // first cell of this instance; of the launch's first instance (field output)
    float4* kout;

    // fb_: first cell of the launch's first instance; a field evaluation writes
    // fout[i - fb_], so a launch over several instances fills [instances][N]
    __device__ __forceinline__ void init(const Buffers& Bf, const StageArgs& A, const InstState& st,
                                         const InstParams& ip, const StageScalars& sc, long long cb_,
                                         long long fb_) {
        nm = NM == 1 ? 1 : A.nmodes;
#pragma unroll
        for (int q = 0; q < NM; q++) {
            G[q] = sc.gamma[q];
            bs[q] = (float)ip.brms_scale[q];
            on[q] = q < nm && ip.cav_on[q] != 0;
        }
        D = sc.drive;
        dt = (float)st.dt;
        bex = (float)ip.bext[0]; bey = (float)ip.bext[1]; bez = (float)ip.bext[2];
        want_demag = A.terms & 1; want_exch = A.terms & 2;
        want_anis = A.terms & 4; want_zee = A.terms & 8; want_cav = A.terms & 16;
        field_only = A.field_only != 0;
        K = A.kind; s = A.stage; mode = A.mode;
        cb = cb_;
        fb = fb_;
        const int k1slot = st.k1slot;
        kout = K == KIND_RK4 ? (s < 3 ? Bf.k[s] : nullptr)
                             : (s < 6 ? Bf.k[s == 0 ? k1slot : s] : Bf.k[k1slot == 0 ? 6 : 0]);
    }

    // (Bx, By, Bz) holds demag + exchange on entry.  MID: a stage that stores
    // its torque and is not the last of its step, with every field term on
    // (all but one launch of a step): none of the checks below is made per cell
    template <bool REC, bool MID>
    __device__ __forceinline__ void run(const Material& mat, const Buffers& Bf, long long i, float4 m, float Bx,
                                        float By, float Bz, Sum3 (&xacc)[NM], Sum3 (&macc)[REC ? 3 : 1],
                                        float& emax, bool& bad) const {
        const float Ms = m.w;
        float px_[NM], py_[NM], pz_[NM];
#pragma unroll
        for (int q = 0; q < NM; q++) px_[q] = py_[q] = pz_[q] = 0.f;
        if (Ms > 0.f) {
            if ((MID || want_anis) && mat.two_ku != 0.f) {
                float mu = m.x * mat.u[0] + m.y * mat.u[1] + m.z * mat.u[2];
                float f = mat.two_ku * __fdividef(mu, Ms);
                Bx += f * mat.u[0]; By += f * mat.u[1]; Bz += f * mat.u[2];
            }
            if (MID || want_zee) { Bx += bex; By += bey; Bz += bez; }
#pragma unroll
            for (int q = 0; q < NM; q++) {
                // the excitation (Appendix C) uses the map of mode 0
                if (!(on[q] || (q == 0 && D != 0.f))) continue;
                if (Bf.prof[q]) {
                    float4 p = __ldg(Bf.prof[q] + (i - cb));
                    px_[q] = bs[q] * p.x; py_[q] = bs[q] * p.y; pz_[q] = bs[q] * p.z;
                } else {
                    py_[q] = bs[q];
                }
                if (on[q] && (MID || want_cav)) { Bx += G[q] * px_[q]; By += G[q] * py_[q]; Bz += G[q] * pz_[q]; }
                if (q == 0 && (MID || want_zee)) { Bx += D * px_[0]; By += D * py_[0]; Bz += D * pz_[0]; }
            }
        }
        if (!MID && field_only) {
            Bf.fout[i - fb] = make_float4(Bx, By, Bz, 0.f);
            return;
        }
        float cx = m.y * Bz - m.z * By, cy = m.z * Bx - m.x * Bz, cz = m.x * By - m.y * Bx;
        float dx = m.y * cz - m.z * cy, dy = m.z * cx - m.x * cz, dz = m.x * cy - m.y * cx;
        float4 kk = make_float4(mat.pre * (cx + mat.alpha * dx), mat.pre * (cy + mat.alpha * dy),
                                mat.pre * (cz + mat.alpha * dz), 0.f);
        if (!(Ms > 0.f)) kk = make_float4(0.f, 0.f, 0.f, 0.f);
        // a NaN or infinite component makes the sum non-finite (so does a
        // component sum beyond the float range, itself an overflowing torque)
        if (!(fabsf(kk.x + kk.y + kk.z) <= 3.0e38f)) bad = true;
        float4 mx = m;   // m used for the coupling sums of this launch
        float4 mrec = m; // state being accepted (recorded spatial average)
        if (MID) {
            kout[i] = kk;
        } else if (K == KIND_RK4) {
            if (s < 3) {
                kout[i] = kk;
            } else {
                float4 m0 = Bf.m[0][i];
                float4 k0 = Bf.k[0][i], k1 = Bf.k[1][i], k2 = Bf.k[2][i];
                float h = dt * (1.f / 6.f);
                float4 mn;
                mn.x = m0.x + h * (k0.x + 2.f * k1.x + 2.f * k2.x + kk.x);
                mn.y = m0.y + h * (k0.y + 2.f * k1.y + 2.f * k2.y + kk.y);
                mn.z = m0.z + h * (k0.z + 2.f * k1.z + 2.f * k2.z + kk.z);
                float r2 = mn.x * mn.x + mn.y * mn.y + mn.z * mn.z;
                float inv = (Ms > 0.f && r2 > 0.f) ? rsqrtf(r2) : 0.f;
                mn.x *= inv; mn.y *= inv; mn.z *= inv;
                mn.w = m0.w;
                Bf.m[0][i] = mn;
                if (mode == CAV_P) mx = mn;
                mrec = mn;
            }
        } else {
            kout[i] = kk;
            if (s == 6) {
                float4 e = Bf.e6[i];
                float c7 = c_ef[6] * dt;
                float exx = e.x + c7 * kk.x, eyy = e.y + c7 * kk.y, ezz = e.z + c7 * kk.z;
                const float en = sqrtf(exx * exx + eyy * eyy + ezz * ezz);
                if (!(en <= 3.0e38f)) bad = true;    // fmaxf would drop a NaN
                emax = fmaxf(emax, en);
            }
        }
        // the coupling sums: m . B_rms,q in FP32, its product with Ms exact
#pragma unroll
        for (int q = 0; q < NM; q++)
            if (on[q]) sum3_add_product(xacc[q], Ms, mx.x * px_[q] + mx.y * py_[q] + mx.z * pz_[q]);
        if constexpr (REC) {
            if (Ms > 0.f) { sum3_add(macc[0], mrec.x); sum3_add(macc[1], mrec.y); sum3_add(macc[2], mrec.z); }
        }
    }
};

// Factor of the Appendix C excitation at this launch's stage time (simulation
// time t + c_s dt): drv_amp sinc(drv_wcut (t - drv_t0)), sinc(0) = 1.
static __device__ double drive_factor(const StageArgs& A, const InstParams& ip, const InstState& st) {
    if (!ip.drv_on) return 0.0;
    const double ts = st.t + (A.field_only ? 0.0 : c_cd[A.kind][A.stage] * st.dt);
    const double x = ip.drv_wcut * (ts - ip.drv_t0);
    return ip.drv_amp * (x == 0.0 ? 1.0 : sin(x) / x);
}

// Whether this is the last stage of a step.
__device__ __forceinline__ bool stage_last(const StageArgs& A) { return A.stage == (A.kind == KIND_RK4 ? 3 : 6); }

// Whether a launch records the spatial average of the state being accepted:
// the last stage of a step with recording on (stage k).
__device__ __forceinline__ bool stage_records(const StageArgs& A, int k) {
    return A.record > 0 && k == (A.kind == KIND_RK4 ? 3 : 6);
}

// All partials of instance b of stage k reduced in a fixed order by this
// block, then the scalar work of that stage, by warp 0: on return f holds the
// lane's mode.  trig as for StageFinish::finish, in shared memory, written by
// other warps before the call.
static __device__ __forceinline__ void finish_instance(const Plan& P, const Material& mat, const Buffers& Bf,
                                                       const StageArgs& A, int b, int k, StageFinish& f,
                                                       float4* s_red, float* s_redf,
                                                       const double (*trig)[MAX_MODES]) {
    const int n = A.nparts;
    const long long pb = (long long)b * n;
    const bool rec = stage_records(A, k), dp_last = A.kind == KIND_DP45 && k == 6;
    const InstParams& ip = Bf.ip[b];
    InstState& st = Bf.st[b];
    double msum[3] = {0.0, 0.0, 0.0}, x = 0.0;
    float em = 0.f;
    const long long ms = (long long)P.B * n;
    const Sum3 z3 = {0.f, 0.f, 0.f};
    if (A.nmodes == 1 && !rec) {
        Sum3 v[1] = {z3};
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
            sum3_merge(v[0], sum3_unpack(__ldcg(Bf.xpart + pb + r)));
            if (dp_last) em = fmaxf(em, __ldcg(Bf.epart + pb + r));
        }
        if (threadIdx.x < 32) f.load(A, k, ip, st);
        block_reduce<1>(v, em, dp_last, s_red, s_redf);
        x = sum3_value(v[0]);
    } else {
        Sum3 v[MAX_MODES + 3];
#pragma unroll
        for (int q = 0; q < MAX_MODES + 3; q++) v[q] = z3;
        for (int r = threadIdx.x; r < n; r += blockDim.x) {
#pragma unroll
            for (int q = 0; q < MAX_MODES; q++)
                if (q < A.nmodes) sum3_merge(v[q], sum3_unpack(__ldcg(Bf.xpart + q * ms + pb + r)));
            if (dp_last) em = fmaxf(em, __ldcg(Bf.epart + pb + r));
            if (rec)
                for (int c = 0; c < 3; c++)
                    sum3_merge(v[MAX_MODES + c], sum3_unpack(__ldcg(Bf.mpart + 3 * (pb + r) + c)));
        }
        if (threadIdx.x < 32) f.load(A, k, ip, st);
        block_reduce<MAX_MODES + 3>(v, em, dp_last, s_red, s_redf);
        if (threadIdx.x < 32) {
            // lane q takes mode q's sum, lane 0 also the average's
            if (rec)
                for (int c = 0; c < 3; c++) msum[c] = sum3_value(v[MAX_MODES + c]);
            Sum3 own = v[0];
#pragma unroll
            for (int q = 0; q < MAX_MODES; q++) {
                Sum3 w;
                w.h = __shfl_sync(0xffffffffu, v[q].h, 0);
                w.m = __shfl_sync(0xffffffffu, v[q].m, 0);
                w.l = __shfl_sync(0xffffffffu, v[q].l, 0);
                if (threadIdx.x == q) own = w;
            }
            x = sum3_value(own);
        }
    }
    if (threadIdx.x < 32) {
        em = __shfl_sync(0xffffffffu, em, 0);
        f.finish(mat, A, k, ip, st, x, em, Bf.hist + (long long)b * Bf.hcap, Bf.hcap, Bf.flags, msum,
                 rec ? Bf.mhist + 4LL * b * Bf.hcap : nullptr, trig);
    }
}

// exp(sign kappa t), sin and cos of omega t of mode q at cavity time t.
static __device__ __noinline__ void mode_trig(const InstParams& ip, int q, double sign, double t,
                                              double (*trig)[MAX_MODES]) {
    double sn, cs;
    sincos(ip.wc[q] * t, &sn, &cs);
    trig[0][q] = exp(sign * ip.kappa[q] * t);
    trig[1][q] = sn;
    trig[2][q] = cs;
}

// alpha_q of the second Dormand-Prince stage of an attempt that kept its first
// one, at the step length now in use (the caller or a horizon may have changed
// it since the last attempt); its real part is returned.  Out of line: inlined
// it cost every stage of a 32x32 film 0.3 us (3.54 against 3.66 ms per 50 RK4
// steps, which never take it).
static __device__ __noinline__ double kept_stage2(InstState& s, int q) {
    const double w = s.dt * c_ad[1][1][0];
    const double a = s.a_re[q] + w * s.ka_re[q][0];
    s.as_re[q] = a;
    s.as_im[q] = s.a_im[q] + w * s.ka_im[q][0];
    return a;
}

// The scalar block of instance b in an x forward (one extra block per
// instance, running beside the row blocks, which need none of what it writes):
// the scalar work the previous stage left (A.fin_prev), then Gamma_k and the
// excitation of this stage for the x inverse that follows.  So neither the
// end of one x inverse nor the start of the next waits for FP64 arithmetic
// (P-mode: an exponential and a sine of each mode in every block, 9 us of a
// 17 us x inverse of a 50^3 sphere with two modes).
static __device__ __noinline__ void scalar_block(const Plan& P, const Material& mat, const Buffers& Bf,
                                                 const StageArgs& A, int b, float4* s_red, float* s_redf) {
    __shared__ double s_end[3][MAX_MODES], s_now[3][MAX_MODES];
    const InstParams& ip = Bf.ip[b];
    const InstState& st = Bf.st[b];
    // a Dormand-Prince stage 1 that was skipped (kept from the last attempt)
    // has nothing to finish
    const bool kept = A.kind == KIND_DP45 && A.fin_prev == 0 && st.have_k1;
    const bool fin = A.fin_prev >= 0 && !kept;
    const bool step_end = fin && A.kind == KIND_RK4 && A.fin_prev == 3;
    const double dt = st.dt;
    const double t_end = st.tcav + (step_end ? dt : 0.0);
    const double t_now = t_end + (A.field_only ? 0.0 : c_cd[A.kind][A.stage] * dt);
    if (threadIdx.x >= 32 && threadIdx.x < 32 + A.nmodes && A.mode == CAV_P) {
        // beside the loads and the reduction of warp 0
        const int q = threadIdx.x - 32;
        if (ip.cav_on[q]) {
            if (step_end) mode_trig(ip, q, 1.0, t_end, s_end);
            mode_trig(ip, q, -1.0, t_now, s_now);
        }
    }
    __syncthreads();        // (and every thread has read the state that warp 0 changes)
    StageFinish f;
    f.ar = 0.0;
    if (fin) finish_instance(P, mat, Bf, A, b, A.fin_prev, f, s_red, s_redf, s_end);
    if (threadIdx.x >= 32) return;
    __syncwarp();
    const int q = threadIdx.x;
    if (q < A.nmodes) {
        float G = 0.f;
        if (ip.cav_on[q]) {
            if (A.mode == CAV_P) {
                G = (float)gamma_p(ip, st, q, s_now[0][q], s_now[1][q], s_now[2][q], mat.hbar);
            } else {
                // (field only, or the first stage of a call: alpha itself)
                G = 2.f * (float)(fin ? f.ar : kept ? kept_stage2(Bf.st[b], q) : st.a_re[q]);
            }
        }
        Bf.sc[b].gamma[q] = G;
    }
    if (q == MAX_MODES) Bf.sc[b].drive = (float)drive_factor(A, ip, st);
}

// The scalar work of this stage, by the last x inverse block to finish.
static __device__ __noinline__ void finish_here(const Plan& P, const Material& mat, const Buffers& Bf,
                                                const StageArgs& A, int b, float4* s_red, float* s_redf) {
    __shared__ double s_end[3][MAX_MODES];
    if (threadIdx.x >= 32 && threadIdx.x < 32 + A.nmodes && A.mode == CAV_P && stage_last(A)) {
        const int q = threadIdx.x - 32;
        const InstState& st = Bf.st[b];
        if (Bf.ip[b].cav_on[q]) mode_trig(Bf.ip[b], q, 1.0, st.tcav + st.dt, s_end);
    }
    __syncthreads();
    StageFinish f;
    finish_instance(P, mat, Bf, A, b, A.stage, f, s_red, s_redf, s_end);
}

// End of an x inverse block: its partials of X_k, of the DP45 error (last
// stage) and of the recorded average.  With A.fin_here the last block of the
// instance to arrive finishes the stage; otherwise the scalar block of the
// next x forward does.  `part` = this block's index among A.nparts.
template <bool REC, int NM>
static __device__ __forceinline__ void stage_epilogue(const Plan& P, const Material& mat, const Buffers& Bf,
                                                      const StageArgs& A, int b, int part, const Sum3 (&xacc)[NM],
                                                      float emax, bool bad, float4* s_red, float* s_redf, int* s_last,
                                                      const Sum3* macc) {
    // RK4: a non-finite torque is an error.  DP45: it marks the attempt, which
    // is then rejected with the smallest step factor (an overflowing trial
    // step); a state that stays non-finite ends in step-size underflow.
    if (bad) {
        if (A.kind == KIND_DP45) atomicOr(&Bf.st[b].poison, 1);
        else atomicOr(Bf.flags, FLAG_NAN);
    }
    const int nparts = A.nparts;
    const bool dp_last = A.kind == KIND_DP45 && A.stage == 6;
    constexpr int NQ = NM + (REC ? 3 : 0);
    Sum3 v[NQ];
#pragma unroll
    for (int q = 0; q < NM; q++) v[q] = xacc[q];
    if constexpr (REC)
        for (int c = 0; c < 3; c++) v[NM + c] = macc[c];
    block_reduce<NQ>(v, emax, dp_last, s_red, s_redf);
    const long long pb = (long long)b * nparts;
    if (threadIdx.x == 0) {
        const int nm = NM == 1 ? 1 : A.nmodes;
#pragma unroll
        for (int q = 0; q < NM; q++)
            if (q < nm) Bf.xpart[((long long)q * P.B + b) * nparts + part] = sum3_pack(v[q]);
        if (dp_last) Bf.epart[pb + part] = emax;
        if constexpr (REC)
            for (int c = 0; c < 3; c++) Bf.mpart[3 * (pb + part) + c] = sum3_pack(v[NM + c]);
        if (A.fin_here) {
            __threadfence();
            unsigned prev = atomicAdd(Bf.counter + b, 1u);
            *s_last = prev == (unsigned)(nparts - 1);
        }
    }
    if (!A.fin_here) return;
    __syncthreads();
    if (!*s_last) return;
    __threadfence();
    if (threadIdx.x == 0) Bf.counter[b] = 0u;
    finish_here(P, mat, Bf, A, b, s_red, s_redf);
}

}  // namespace mq
