// The proximal map of alpha (R3 + delta_{>=0}) with all three terms of Eq.
// (reg-tv-l1-one): TV of every species, l1, and TV of every pulse image
// (S c)^n -- the lambda_3 term -- by Algorithm 2 on the stacked operator
//   L v = [ lam_tv D v_p (p < P) ;  lam_l1 v ;  lam_b D (S v)^n (n < N) ],
// with D the 3D forward differences (zero across the far faces) and
// (S v)^n[j] = sum_p S[m(n)][p][j] v_p[j], m(n) = n mod pulses_per_cycle.
// The prox of Eq. (prox) includes the nonnegativity indicator, and Eq.
// (prox-dual) keeps the matching constraint z - L^T u >= 0, so the dual is
// min over |u| <= alpha of 1/2 ||max(z - L^T u, 0)||^2 and the projected
// primal point enters every step, from u = r = 0:
//   w   = max(z - L^T r, 0)
//   u_i = clamp(r + step2 L w, -alpha, alpha)
//   r   = u_i + beta_i (u_i - u_{i-1})          (Beck-Teboulle beta_i)
// and x = max(z - L^T u, 0).
//
// Pulses of one switching state m share the image S_m v, so their duals
// receive the same gradient from the same start and stay equal; one dual per
// state, entering L^T with the state's pulse count C_m, gives Algorithm 2's
// iterates with 3 Q instead of 3 N pulse-image components.
//
// The switching weights depend on the depth only, so L^T of the dual needs no
// more than four sums per voxel and species over all of the voxel's entries,
//   e0, e1 = lam_tv r_tv,c + lam_b sum_m C_m S[m][p][j] r_m,c   (c = y, x)
//   e2     = the same for c = z with the weights of depth j + 1
//   f      = lam_l1 r_l1 - e0 - e1 - (e2 with the weights of depth j),
//   (L^T r)_p[i] = f[i] + e0[i - y] + e1[i - x] + e2[i - 1],
// which the thread that updates the voxel's dual has in registers.  And r is
// not stored: r = u_i + beta_i (u_i - u_{i-1}) of the two dual iterates is formed
// again where it is read, and u_{i+1} overwrites u_{i-1}.  So an iteration is
// two voxel-parallel kernels, w from the sums (6 P volumes), then the dual step
// (2 nd read, nd written, nd = 4 P + 3 Q, and 5 P), where a kernel for L^T of all
// entries and a dual step with r stored moved 5 nd + 3 P.  Both are bound by
// memory; a thread issues the loads of a group of states before their
// arithmetic.  P = 3, Q = 10: 159 volumes instead of 219 per iteration;
// 10 iterations at 96 x 80 x 77 729 us instead of 1010, at 128 x 128 x 96 1826
// instead of 2593 (5.5 TB/s).
// The first iteration reads no dual (r = u = 0).  Scratch (w, the sums and two
// dual iterates) is the handle's.
#include <algorithm>
#include <cmath>

#include "swopt_internal.cuh"

namespace swopt {
namespace {

constexpr int kJointBlock = 256;
constexpr int kJointMaxSpecies = 8;
constexpr int kStateChunk = 4;  // switching states whose loads are issued together


struct JointArgs {
    int P, Q, Y, X, Z;
    const float* Sm;   // [Q][P][Z] switching weights of the states
    const float* Cmf;  // [Q] pulses per state
    float lam_tv, lam_l1, lam_b;
};

// Voxel i = (y X + x) Z + j of a volume with fewer than 2^31 voxels.
struct Vox {
    int y, x, j;
    __device__ __forceinline__ Vox(unsigned i, const JointArgs& a)
    {
        const unsigned t = i / (unsigned)a.Z;
        j = (int)(i - t * (unsigned)a.Z);
        y = (int)(t / (unsigned)a.X);
        x = (int)(t - (unsigned)y * (unsigned)a.X);
    }
};

// out = max(z - L^T r, 0) from the sums e [4][NP][L] (f, e0, e1, e2; null:
// r = 0), one thread per voxel, all NP species.  z and out may be the same
// array: each thread reads z at its voxel before writing there.
template <int NP>
__global__ void __launch_bounds__(kJointBlock)
    joint_primal_kernel(const JointArgs a, const float* z, const float* e, float* out)
{
    grid_dependency();
    const unsigned L = (unsigned)a.Y * a.X * a.Z;
    const size_t Ls = L, sy = (size_t)a.X * a.Z, sx = (size_t)a.Z;
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < L; i += gridDim.x * blockDim.x) {
        const Vox q(i, a);
        float v[NP], t[NP][4];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            v[p] = z[(size_t)p * Ls + i];
#pragma unroll
            for (int c = 0; c < 4; ++c) t[p][c] = 0.f;
            if (e) {
                const float* ep = e + (size_t)p * Ls + i;
                t[p][0] = load_produced(ep);
                if (q.y > 0) t[p][1] = load_produced(ep + NP * Ls - sy);
                if (q.x > 0) t[p][2] = load_produced(ep + 2 * NP * Ls - sx);
                if (q.j > 0) t[p][3] = load_produced(ep + 3 * NP * Ls - 1);
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p)
            out[(size_t)p * Ls + i] =
                fmaxf(v[p] - ((t[p][0] + t[p][1]) + (t[p][2] + t[p][3])), 0.f);
    }
}

// One dual step of every entry of a voxel.  ua: u_i; ub: u_{i-1}, overwritten
// with u_{i+1} = clamp(r_i + step2 L w, -alpha, alpha); e: the sums of r_{i+1}
// (beta 0: of u_{i+1}).  done: dual iterates that exist (0: u = 0, 1: u_{i-1} = 0).
template <int NP>
__global__ void __launch_bounds__(kJointBlock, NP <= 4 ? 3 : 2)
    joint_dual_kernel(const JointArgs a, const float* w, const float* ua, float* ub, float* e, float step2, float alpha, float beta_prev,
                      float beta, int done)
{
    grid_dependency();
    const unsigned L = (unsigned)a.Y * a.X * a.Z;
    const size_t Ls = L, sy = (size_t)a.X * a.Z, sx = (size_t)a.Z;
    const size_t ol = (size_t)NP * 3 * Ls, ob = ol + (size_t)NP * Ls;
    // the step of one entry: its loaded u_i and u_{i-1}, and L w there; returns r_{i+1}
    auto step = [&](size_t at, float u, float up, float lw) -> float {
        const float r = fmaf(beta_prev, u - up, u);
        const float v = fminf(fmaxf(fmaf(step2, lw, r), -alpha), alpha);
        ub[at] = v;
        return fmaf(beta, v - u, v);
    };
    for (unsigned i = blockIdx.x * blockDim.x + threadIdx.x; i < L; i += gridDim.x * blockDim.x) {
        const Vox q(i, a);
        const bool hy = q.y + 1 < a.Y, hx = q.x + 1 < a.X, hz = q.j + 1 < a.Z;
        // w at the voxel and its three forward neighbours (0 past the far faces)
        float w0[NP], wy[NP], wx[NP], wz[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const float* wp = w + (size_t)p * Ls + i;
            w0[p] = load_produced(wp);
            wy[p] = hy ? load_produced(wp + sy) : 0.f;
            wx[p] = hx ? load_produced(wp + sx) : 0.f;
            wz[p] = hz ? load_produced(wp + 1) : 0.f;
        }
        float f[NP], e0[NP], e1[NP], e2[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            const size_t at[4] = {(size_t)p * 3 * Ls + i, (size_t)p * 3 * Ls + Ls + i,
                                  (size_t)p * 3 * Ls + 2 * Ls + i, ol + (size_t)p * Ls + i};
            float u[4], up[4];
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                u[c] = done > 0 ? load_produced(ua + at[c]) : 0.f;
                up[c] = done > 1 ? ub[at[c]] : 0.f;
            }
            const float lw[4] = {hy ? a.lam_tv * (wy[p] - w0[p]) : 0.f,
                                 hx ? a.lam_tv * (wx[p] - w0[p]) : 0.f,
                                 hz ? a.lam_tv * (wz[p] - w0[p]) : 0.f, a.lam_l1 * w0[p]};
            e0[p] = a.lam_tv * step(at[0], u[0], up[0], lw[0]);
            e1[p] = a.lam_tv * step(at[1], u[1], up[1], lw[1]);
            e2[p] = a.lam_tv * step(at[2], u[2], up[2], lw[2]);
            f[p] = a.lam_l1 * step(at[3], u[3], up[3], lw[3]) - e2[p];
        }
        for (int m0 = 0; m0 < a.Q; m0 += kStateChunk) {
            float u[kStateChunk][3], up[kStateChunk][3];
#pragma unroll
            for (int c = 0; c < kStateChunk; ++c) {
                const size_t at = ob + (size_t)(m0 + c) * 3 * Ls + i;
                const bool in = m0 + c < a.Q;
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    u[c][k] = in && done > 0 ? load_produced(ua + at + k * Ls) : 0.f;
                    up[c][k] = in && done > 1 ? ub[at + k * Ls] : 0.f;
                }
            }
#pragma unroll
            for (int c = 0; c < kStateChunk; ++c) {
                const int m = m0 + c;
                if (m >= a.Q) break;
                const float* s = a.Sm + (size_t)m * NP * a.Z + q.j;
                float sj[NP], sn[NP];
                float b0 = 0.f, by = 0.f, bx = 0.f, bz = 0.f;
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    sj[p] = __ldg(s + (size_t)p * a.Z);
                    sn[p] = hz ? __ldg(s + (size_t)p * a.Z + 1) : 0.f;
                    b0 = fmaf(sj[p], w0[p], b0);
                    by = fmaf(sj[p], wy[p], by);
                    bx = fmaf(sj[p], wx[p], bx);
                    if (hz) bz = fmaf(sn[p], wz[p], bz);
                }
                const size_t at = ob + (size_t)m * 3 * Ls + i;
                const float g = __ldg(a.Cmf + m) * a.lam_b;
                const float d0 = g * step(at, u[c][0], up[c][0], hy ? a.lam_b * (by - b0) : 0.f);
                const float d1 = g * step(at + Ls, u[c][1], up[c][1], hx ? a.lam_b * (bx - b0) : 0.f);
                const float d2 =
                    g * step(at + 2 * Ls, u[c][2], up[c][2], hz ? a.lam_b * (bz - b0) : 0.f);
#pragma unroll
                for (int p = 0; p < NP; ++p) {
                    e0[p] = fmaf(sj[p], d0, e0[p]);
                    e1[p] = fmaf(sj[p], d1, e1[p]);
                    e2[p] = fmaf(sn[p], d2, e2[p]);
                    f[p] = fmaf(-sj[p], d2, f[p]);
                }
            }
        }
#pragma unroll
        for (int p = 0; p < NP; ++p) {
            float* ep = e + (size_t)p * Ls + i;
            ep[0] = f[p] - e0[p] - e1[p];
            ep[NP * Ls] = e0[p];
            ep[2 * NP * Ls] = e1[p];
            ep[3 * NP * Ls] = e2[p];
        }
    }
}

// Algorithm 2 for NP species (see the file comment).
template <int NP>
swopt_status joint_prox_np(swopt_handle* h, const JointArgs& a, const float* z, float* x, float alpha,
                           int iters, float step2, int momentum, float* w, float* u0, float* u1,
                           float* e, cudaStream_t st)
{
    const size_t L = (size_t)h->Y * h->X * h->Z;
    int sms = 0;
    SW_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    const int grid = (int)std::min<size_t>((size_t)grid_for(L, kJointBlock), (size_t)sms * 16);
    double t = 1.0, prev = 0.0;
    for (int it = 0; it < iters; ++it) {
        const double t1 = 0.5 * (1.0 + std::sqrt(1.0 + 4.0 * t * t));
        const double b = momentum == SWOPT_MOMENTUM_BECK_TEBOULLE ? (t - 1.0) / t1
                         : momentum == SWOPT_MOMENTUM_PAPER_PRINTED ? (t - 1.0) / (t + 1.0)
                                                                    : 0.0;
        t = t1;
        SW_CUDA(launch_pdl(joint_primal_kernel<NP>, grid, kJointBlock, 0, st, a, z,
                           it == 0 ? (const float*)nullptr : (const float*)e, w));
        SW_LAUNCHED(h);
        // the sums of the last iteration are those of u_K, for the output
        SW_CUDA(launch_pdl(joint_dual_kernel<NP>, grid, kJointBlock, 0, st, a, (const float*)w,
                           (const float*)u0, u1, e, step2, alpha, (float)prev,
                           it + 1 == iters ? 0.f : (float)b, it));
        SW_LAUNCHED(h);
        std::swap(u0, u1);
        prev = b;
    }
    SW_CUDA(launch_pdl(joint_primal_kernel<NP>, grid, kJointBlock, 0, st, a, z,
                       iters == 0 ? (const float*)nullptr : (const float*)e, x));
    SW_LAUNCHED(h);
    return SWOPT_OK;
}

}  // namespace

size_t joint_dual_floats(const swopt_handle* h)
{
    const size_t L = (size_t)h->Y * h->X * h->Z;
    return (size_t)h->P * 4 * L + (size_t)h->Q * 3 * L;
}

double joint_step_bound(const swopt_handle* h, double lambda_tv, double lambda_l1,
                        double lambda_b)
{
    // ||L||^2 <= 12 lam_tv^2 + lam_l1^2 + 12 lam_b^2 sum_n max_j sum_p S[n][p][j]^2
    // (||D||^2 <= 12 in 3D; |(S_n v)_voxel|^2 <= (sum_p S^2)(sum_p v_p^2) at every voxel)
    double s2 = 0.0;
    for (int m = 0; m < h->Q; ++m) {
        double mx = 0.0;  // max over depths of sum_p S_m[p][j]^2
        for (int j = 0; j < h->Z; ++j) {
            double a = 0.0;
            for (int p = 0; p < h->P; ++p) {
                const double v = h->Sm64[((size_t)m * h->P + p) * h->Z + j];
                a += v * v;
            }
            mx = a > mx ? a : mx;
        }
        s2 += h->Cm[m] * mx;
    }
    return 12.0 * lambda_tv * lambda_tv + lambda_l1 * lambda_l1 + 12.0 * lambda_b * lambda_b * s2;
}

// Algorithm 2 on the stacked L (see the file comment) with caller-given
// scratch: w [P L], the two dual iterates u and r [(4 P + 3 Q) L] each, and the
// sums e [4 P L].  Asynchronous on st.
swopt_status joint_prox_on(swopt_handle* h, const float* z, float* x, double alpha,
                           double lambda_tv, double lambda_l1, double lambda_b, int iters,
                           double step2, int momentum, float* w, float* u, float* r,
                           float* e, cudaStream_t st)
{
    if (h->P > kJointMaxSpecies) {
        set_error("the joint prox supports at most %d species", kJointMaxSpecies);
        return SWOPT_ERR_UNSUPPORTED;
    }
    const size_t L = (size_t)h->Y * h->X * h->Z;
    if (L >= (1ull << 31)) {
        set_error("the joint prox supports volumes below 2^31 voxels");
        return SWOPT_ERR_UNSUPPORTED;
    }
    JointArgs a;
    a.P = h->P;
    a.Q = h->Q;
    a.Y = h->Y;
    a.X = h->X;
    a.Z = h->Z;
    a.Sm = h->Sm;
    a.Cmf = h->Cmf;
    a.lam_tv = (float)lambda_tv;
    a.lam_l1 = (float)lambda_l1;
    a.lam_b = (float)lambda_b;
    switch (a.P) {
#define SWOPT_JOINT_CASE(n)                                                                     \
    case n:                                                                                     \
        return joint_prox_np<n>(h, a, z, x, (float)alpha, iters, (float)step2, momentum, w, u, r, e, \
                                st);
        SWOPT_JOINT_CASE(1)
        SWOPT_JOINT_CASE(2)
        SWOPT_JOINT_CASE(3)
        SWOPT_JOINT_CASE(4)
        SWOPT_JOINT_CASE(5)
        SWOPT_JOINT_CASE(6)
        SWOPT_JOINT_CASE(7)
        SWOPT_JOINT_CASE(8)
#undef SWOPT_JOINT_CASE
    }
    set_error("the joint prox supports 1 to %d species", kJointMaxSpecies);
    return SWOPT_ERR_UNSUPPORTED;
}

swopt_status ensure_joint_buffers(swopt_handle* h)
{
    const size_t nu = joint_dual_floats(h);
    if (!h->jw) SW_CUDA(cudaMalloc((void**)&h->jw, sizeof(float) * nc_of(h)));
    if (!h->ju) SW_CUDA(cudaMalloc((void**)&h->ju, sizeof(float) * nu));
    if (!h->jr) SW_CUDA(cudaMalloc((void**)&h->jr, sizeof(float) * nu));
    if (!h->je) SW_CUDA(cudaMalloc((void**)&h->je, sizeof(float) * 4 * nc_of(h)));
    return SWOPT_OK;
}

}  // namespace swopt

using namespace swopt;

extern "C" {

swopt_status swopt_prox_joint(swopt_handle* h, const float* z_dev, float* x_dev, double alpha,
                              double lambda_tv, double lambda_l1, double lambda_b, int iters,
                              double step2, void* stream)
{
    clear_error();
    if (!h) {
        set_error("null handle");
        return SWOPT_ERR_INVALID_ARG;
    }
    if (!z_dev || !x_dev || !std::isfinite(alpha) || alpha < 0.0 || !std::isfinite(lambda_tv) ||
        lambda_tv < 0.0 || !std::isfinite(lambda_l1) || lambda_l1 < 0.0 ||
        !std::isfinite(lambda_b) || lambda_b < 0.0 || iters < 0 ||
        (iters > 0 && (!std::isfinite(step2) || !(step2 > 0.0)))) {
        set_error("invalid joint-prox arguments");
        return SWOPT_ERR_INVALID_ARG;
    }
    if (h->P > kJointMaxSpecies) {
        set_error("the joint prox supports at most %d species", kJointMaxSpecies);
        return SWOPT_ERR_UNSUPPORTED;
    }
    SW_TRY(ensure_joint_buffers(h));
    return joint_prox_on(h, z_dev, x_dev, alpha, lambda_tv, lambda_l1, lambda_b, iters, step2,
                         SWOPT_MOMENTUM_BECK_TEBOULLE, h->jw, h->ju, h->jr, h->je,
                         (cudaStream_t)stream);
}

double swopt_prox_joint_step_bound(swopt_handle* h, double lambda_tv, double lambda_l1,
                                   double lambda_b)
{
    if (!h) return 0.0;
    return joint_step_bound(h, lambda_tv, lambda_l1, lambda_b);
}

}  // extern "C"
