// The TV prox (Algorithm 2) and the FISTA step after it with the whole state
// on the chip, for volumes that fit: one cooperative launch, every inner
// iteration without a pass over memory.
//
// A block owns TY x TX columns over all depths.  A warp owns one x column and
// marches along y, its lanes along z (depth 32 v + lane, v < V).  With the march
// in y and the depths in a warp, almost everything a point needs is its own
// thread's: the duals r0 (along y) and r2 (along z, neighbours by shuffle) stay
// in registers, row by row; only r1 (along x) and two rows of x = z - D^T r are
// read by the neighbouring warp, through shared memory, which also holds u.  One
// barrier per row orders them:
//   step s:  x of row s (reads r of row s and r0 of row s - 1, all old) -> shared
//            barrier
//            dual step of row s - 1 (reads x of rows s - 1 and s, and of the
//            column to the right), in place.
// The ghosts of a block are its neighbours' first and last rows and columns of
// r, published in global memory (two buffers by parity of the iteration) and
// announced by a per-block counter: a block waits for the six neighbours that
// it exchanges with, not for the whole grid.  One more row step and one more
// warp recompute x on the row below and the column to the right.
//
// Volumes that hold more than the chip does at once, but whose species fit one
// by one, take their species in rounds.  The arithmetic per entry is that of
// fgp_iter_kernel.
//
// Bound by the latency of the row steps (one block of 17 warps per SM on the
// largest volume) and the exchange, about 2.5 us per iteration.  10 iterations,
// us, here / as before (fgp_coop_kernel or fgp_tile_kernel): 3 x 128^2 x 96 305 /
// 592, 2 x 64^3 67 / 96, 3 x 64^2 x 123 148 / 287, 2 x 16^2 x 24 31 / 54.
// Registers decide: four depths a lane with 72 registers (540 B of spills) ran
// at 95 us where 168 registers take 61 (2 x 48^2 x 117); tiles of other shapes
// that fit were within 3% or slower.
#include <algorithm>
#include <cmath>

#include "swopt_internal.cuh"

namespace swopt {
namespace {

constexpr int kMaxBetas = 64;
constexpr uint32_t kFlagPolls = 1u << 25;  // x 32 ns back-off: about a second

struct March {
    const float* z;      // prox input [P][Y][X][Z]
    float* pub[2];       // published duals [3][P][Y][X][Z], by parity
    int P, Y, X, Z;
    size_t L;            // P Y X Z
    int TY, TX, tilesY, tilesX;
    int SP, rounds;      // species per round
    float tau;
    int iters;
    int inner_momentum;
    float beta[kMaxBetas];  // inner momentum of the first iterations
    int mode;            // 0: out = z - D^T u;  1: FISTA finish
    float* out;
    float* c;
    float* xi;
    float* delta;        // optional (mode 1)
    double* scal;        // FISTA t_k, beta_k (mode 1)
    int momentum;
    float theta;
    unsigned* bar;       // [2] error, [4] phantom, [5] poll limit, [6] arrivals (see prox.cu)
    unsigned* flags;     // [blocks] iterations finished, over all launches
};

__device__ __forceinline__ double coefficient(double t, double t1, int mode)
{
    if (mode == SWOPT_MOMENTUM_BECK_TEBOULLE) return (t - 1.0) / t1;
    if (mode == SWOPT_MOMENTUM_PAPER_PRINTED) return (t - 1.0) / (t + 1.0);
    return 0.0;
}

__device__ __forceinline__ unsigned load_acquire(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.gpu.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ float clamp_tau(float v, float tau) { return fminf(fmaxf(v, -tau), tau); }

// Most threads of a block, so that the rows' state stays in registers.
__host__ __device__ constexpr int march_threads(int TYT)
{
    return TYT <= 2 ? 1024 : TYT <= 4 ? 832 : TYT <= 6 ? 704 : TYT <= 8 ? 576 : 480;
}

// Blocks of up to 11 warps get a variant of their own for three and four depths
// a lane: 168 registers, where the rows' state would spill.
constexpr int kSmallThreads = 352;

template <int V, int TYT, bool SMALL>
__global__ void __launch_bounds__(SMALL ? kSmallThreads : march_threads(TYT)) fgp_march_kernel(const March a)
{
    extern __shared__ float sm[];
    constexpr int ZS = 32 * V;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int Z = a.Z;
    const size_t L = a.L;
    const int tiles = a.tilesY * a.tilesX;
    const int tx = (int)blockIdx.x % a.tilesX, ty = (int)blockIdx.x / a.tilesX % a.tilesY;
    const int slot = (int)blockIdx.x / tiles;
    const int y0 = ty * a.TY, x0 = tx * a.TX;
    const int ny = min(a.TY, a.Y - y0), nx = min(a.TX, a.X - x0);
    const int gx = x0 + w;
    const bool own = w < nx, ghost_col = w == nx && gx < a.X, active = own || ghost_col;
    const bool ghost_row = y0 + ny < a.Y;
    const bool has_xl = gx > 0, has_xr = gx + 1 < a.X;
    // shared: r1 [TY][TX], u [3][TY][TX], x [3][TX + 1], each ZS floats
    const int plane = a.TY * a.TX * ZS, rs = a.TX * ZS, xs = (a.TX + 1) * ZS;
    const size_t XZ = (size_t)a.X * Z;
    // depth 32 v + lane exists (only the last v can be partial)
    auto in_z = [&](int v) { return v + 1 < V || 32 * (V - 1) + lane < Z; };
    float* s_r1 = sm + lane;
    float* s_u = s_r1 + plane;
    float* s_x = s_u + 3 * plane;
    auto at = [&](int row, int col) { return (row * a.TX + col) * ZS; };

    __shared__ float s_beta;
    __shared__ double s_outer;
    const unsigned base0 = a.flags[blockIdx.x];  // only this block writes it
    if (threadIdx.x == 0) {
        if (a.mode == 1) {
            // Algorithm 1's t_k -> t_{k+1} and beta_k: every block reads t_k, the last
            // one to have done so writes the new scalars
            const double t = *(volatile const double*)a.scal;
            const double t1 = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
            s_outer = coefficient(t, t1, a.momentum);
            unsigned arrived;
            asm volatile("atom.add.acq_rel.gpu.u32 %0, [%1], 1;"
                         : "=r"(arrived) : "l"(a.bar + 6) : "memory");
            if (arrived == gridDim.x - 1) {
                a.bar[6] = 0u;
                a.scal[1] = s_outer;
                a.scal[0] = t1;
            }
        }
    }

    // Waits until the neighbours have finished `target` iterations (bounded: an
    // error is recorded and every later wait returns at once).
    auto wait_for = [&](unsigned target) {
        if (w == 0) {
            // left, right, up, down, down-left, up-right; lane 6: the test hook
            const int dyx[6][2] = {{0, -1}, {0, 1}, {-1, 0}, {1, 0}, {1, -1}, {-1, 1}};
            volatile unsigned* vb = a.bar;
            int nb = -1;
#pragma unroll
            for (int i = 0; i < 6; ++i)
                if (lane == i) {
                    const int ny2 = ty + dyx[i][0], nx2 = tx + dyx[i][1];
                    if (ny2 >= 0 && ny2 < a.tilesY && nx2 >= 0 && nx2 < a.tilesX)
                        nb = slot * tiles + ny2 * a.tilesX + nx2;
                }
            if (lane == 6 && vb[4] != 0u) {
                nb = (int)blockIdx.x;
                target += 1u << 30;  // never reached
            }
            if (nb >= 0 && vb[2] == 0u) {
                uint32_t limit = kFlagPolls;
                if (vb[5] != 0u) limit = vb[5];
                uint32_t polls = 0;
                while ((int)(load_acquire(a.flags + nb) - target) < 0 && vb[2] == 0u) {
                    if (++polls > limit) {
                        atomicExch(&a.bar[2], 1u);
                        break;
                    }
                    if (polls > 256) __nanosleep(32);
                }
            }
            __syncwarp();
        }
        __syncthreads();
    };

    for (int round = 0; round < a.rounds; ++round) {
        const int p = round * a.SP + slot;
        const bool work = p < a.P;  // a last round may leave blocks idle
        const unsigned base = base0 + (unsigned)(round * a.iters);
        // element of column (row, col) of the tile at depth `lane`; rows -1 .. ny and
        // columns -1 .. nx may be asked for where the volume has them
        auto elem = [&](int row, int col) -> size_t {
            return (((size_t)p * a.Y + (y0 + row)) * a.X + (x0 + col)) * Z + lane;
        };
        float r0[TYT + 1][V], r2[TYT + 1][V];
#pragma unroll
        for (int s = 0; s <= TYT; ++s)
#pragma unroll
            for (int v = 0; v < V; ++v) r0[s][v] = r2[s][v] = 0.f;
        if (own)
            for (int s = 0; s < ny; ++s)
#pragma unroll
                for (int v = 0; v < V; ++v) {
                    s_r1[at(s, w) + 32 * v] = 0.f;
                    s_u[at(s, w) + 32 * v] = 0.f;
                    s_u[plane + at(s, w) + 32 * v] = 0.f;
                    s_u[2 * plane + at(s, w) + 32 * v] = 0.f;
                }
        double t = 1.0;
        for (int it = 0; it < a.iters && work; ++it) {
            float beta;
            if (it < kMaxBetas) {
                beta = a.beta[it];
            } else {
                if (threadIdx.x == 0) {
                    if (it == kMaxBetas)  // the recursion up to here
                        for (int i = 0; i < kMaxBetas; ++i) t = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
                    const double t1 = 0.5 * (1.0 + sqrt(1.0 + 4.0 * t * t));
                    s_beta = (float)coefficient(t, t1, a.inner_momentum);
                    t = t1;
                }
                __syncthreads();
                beta = s_beta;
            }
            const bool last = it + 1 == a.iters;
            const float* pr = a.pub[(it + 1) & 1];  // iteration it - 1
            float* pw = a.pub[it & 1];
            // every thread reads ghosts below: the wait's barrier comes first
            wait_for(base + (unsigned)it);
            // Missing neighbours and the far faces read as zero (a dual entry of the last
            // layer stays 0), so the sums below need no conditions.
            const bool old = it > 0;
            auto ghost = [&](int comp, int row, int col, float (&d)[V], bool use) {
                const float* g = pr + (size_t)comp * L + elem(row, col);
#pragma unroll
                for (int v = 0; v < V; ++v) d[v] = use && old && in_z(v) ? __ldcg(g + 32 * v) : 0.f;
            };
            float up[V];  // r0 of the row above
            ghost(0, -1, w, up, active && y0 > 0);
            // ghosts into the registers that hold the own rows' r0 and r2 elsewhere
            if (ghost_col) {
#pragma unroll
                for (int s = 0; s < TYT; ++s) {
                    ghost(0, s, w, r0[s], s < ny);
                    ghost(2, s, w, r2[s], s < ny);
                }
            }
            if (own && ghost_row) {
#pragma unroll
                for (int s = 1; s <= TYT; ++s)
                    if (s == ny) {
                        ghost(0, s, w, r0[s], true);
                        ghost(2, s, w, r2[s], true);
                    }
            }
            // running addresses: z and the published r1 of this column and the one to the left
            const float* zp = a.z + elem(0, w);
            const float* gp = pr + L + elem(0, w);
            const float* sr = s_r1 + w * ZS;   // own r1, row by row
            float* su = s_u + w * ZS;
            float zn[V], bn[V], ln[V], xp[V];
            // what a row needs beside the registers: z, r1 and r1 of the column to the left
            auto fetch = [&](bool in_row) {
                if (own && in_row) {
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        zn[v] = in_z(v) ? __ldg(zp + 32 * v) : 0.f;
                        bn[v] = sr[32 * v];
                    }
                } else {
                    const bool use = own ? ghost_row : ghost_col && in_row;
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        zn[v] = use && in_z(v) ? __ldg(zp + 32 * v) : 0.f;
                        bn[v] = use && old && in_z(v) ? __ldcg(gp + 32 * v) : 0.f;
                    }
                }
                if (w > 0 && in_row) {
#pragma unroll
                    for (int v = 0; v < V; ++v) ln[v] = sr[32 * v - ZS];
                } else {
                    const bool use = old && has_xl && (in_row || ghost_row);
#pragma unroll
                    for (int v = 0; v < V; ++v)
                        ln[v] = use && in_z(v) ? __ldcg(gp - Z + 32 * v) : 0.f;
                }
            };
            if (active) fetch(true);
#pragma unroll
            for (int v = 0; v < V; ++v) xp[v] = 0.f;
#pragma unroll
            for (int s = 0; s <= TYT; ++s) {
                if (s > ny) break;
                float x[V];
                if (active) {
                    float prev[V];  // r2 of the depth above: lane 0 takes it from lane 31 of v - 1
#pragma unroll
                    for (int v = 0; v < V; ++v) prev[v] = __shfl_sync(0xffffffffu, r2[s][v], (lane + 31) & 31);
#pragma unroll
                    for (int v = V - 1; v > 0; --v) prev[v] = lane == 0 ? prev[v - 1] : prev[v];
                    prev[0] = lane == 0 ? 0.f : prev[0];
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const float above = s == 0 ? up[v] : r0[s > 0 ? s - 1 : 0][v];
                        x[v] = zn[v] - (above - r0[s][v] - bn[v] + ln[v] - r2[s][v] + prev[v]);
                    }
                    if (s < ny) {
#pragma unroll
                        for (int v = 0; v < V; ++v) s_x[(s % 3) * xs + w * ZS + 32 * v] = x[v];
                        zp += XZ;
                        gp += XZ;
                        sr += rs;
                        fetch(s + 1 < ny);
                    }
                }
                __syncthreads();
                if (s > 0 && own) {
                    const int row = s > 0 ? s - 1 : 0;
                    float next[V];  // x of the depth below
#pragma unroll
                    for (int v = 0; v < V; ++v) next[v] = __shfl_sync(0xffffffffu, xp[v], (lane + 1) & 31);
#pragma unroll
                    for (int v = 0; v + 1 < V; ++v) next[v] = lane == 31 ? next[v + 1] : next[v];
                    const bool has_yd = s < ny || ghost_row;
                    const float* xr = s_x + (row % 3) * xs + (w + 1) * ZS;
                    float* r1 = su - s_u + s_r1;
                    auto dual = [&](float d, float r, float* u) -> float {
                        const float un = clamp_tau(fmaf(d, 1.0f / 12.0f, r), a.tau);
                        const float n = fmaf(beta, un - *u, un);
                        *u = un;
                        return n;
                    };
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        // no difference past the far faces (also of an infinity or NaN)
                        const float d0 = has_yd ? x[v] - xp[v] : 0.f;
                        const float d1 = has_xr ? xr[32 * v] - xp[v] : 0.f;
                        const float d2 = 32 * v + lane < Z - 1 ? next[v] - xp[v] : 0.f;
                        r0[row][v] = dual(d0, r0[row][v], su + 32 * v);
                        r1[32 * v] = dual(d1, r1[32 * v], su + plane + 32 * v);
                        r2[row][v] = dual(d2, r2[row][v], su + 2 * plane + 32 * v);
                    }
                    if (row == 0 || row == ny - 1 || w == 0 || w == nx - 1) {
                        float* e = pw + elem(row, w);
#pragma unroll
                        for (int v = 0; v < V; ++v)
                            if (in_z(v)) {
                                __stcg(e + 32 * v, last ? su[32 * v] : r0[row][v]);
                                __stcg(e + L + 32 * v, last ? su[plane + 32 * v] : r1[32 * v]);
                                __stcg(e + 2 * L + 32 * v, r2[row][v]);
                            }
                    }
                    su += rs;
                }
#pragma unroll
                for (int v = 0; v < V; ++v) xp[v] = x[v];
            }
            // this block's iteration is published
            __syncthreads();
            if (threadIdx.x == 0)
                asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(a.flags + blockIdx.x),
                             "r"(base + (unsigned)it + 1u)
                             : "memory");
        }
        if (!work) {
            // idle in this round: keep the block's count in step
            if (threadIdx.x == 0)
                asm volatile("st.release.gpu.u32 [%0], %1;" ::"l"(a.flags + blockIdx.x),
                             "r"(base + (unsigned)a.iters)
                             : "memory");
            __syncthreads();
            continue;
        }
        wait_for(base + (unsigned)a.iters);
        // out = z - D^T u, or the end of the FISTA iteration
        const float fb = a.mode == 1 ? (float)s_outer : 0.f;
        const float* pu = a.pub[(a.iters - 1) & 1];
        if (own) {
            // two rows at a time, their reads together
            const bool up_ok = y0 > 0, left = w == 0 && has_xl;
            for (int s0 = 0; s0 < ny; s0 += 2) {
                float zz[2][V], ab[2][V], lf[2][V], cc[2][V];
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        const int s = s0 + h;
                        const bool use = s < ny && in_z(v);
                        const size_t e = elem(s, w) + 32 * v;
                        zz[h][v] = use ? __ldg(a.z + e) : 0.f;
                        cc[h][v] = use && a.mode == 1 ? a.c[e] : 0.f;
                        ab[h][v] = use && s == 0 && up_ok ? __ldcg(pu + elem(-1, w) + 32 * v) : 0.f;
                        lf[h][v] = use && left ? __ldcg(pu + L + elem(s, -1) + 32 * v) : 0.f;
                    }
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int s = s0 + h;
                    if (s >= ny) break;
                    const int o = at(s, w);
                    float u2[V], prev[V];
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        u2[v] = s_u[2 * plane + o + 32 * v];
                        prev[v] = __shfl_sync(0xffffffffu, u2[v], (lane + 31) & 31);
                    }
#pragma unroll
                    for (int v = V - 1; v > 0; --v) prev[v] = lane == 0 ? prev[v - 1] : prev[v];
                    prev[0] = lane == 0 ? 0.f : prev[0];
#pragma unroll
                    for (int v = 0; v < V; ++v) {
                        if (!in_z(v)) continue;
                        const size_t e = elem(s, w) + 32 * v;
                        const float above = s > 0 ? s_u[o - rs + 32 * v] : ab[h][v];
                        const float l = w > 0 ? s_u[plane + o - ZS + 32 * v] : lf[h][v];
                        const float xv = zz[h][v] - (above - s_u[o + 32 * v] - s_u[plane + o + 32 * v] +
                                                     l - u2[v] + prev[v]);
                        if (a.mode == 0) {
                            a.out[e] = xv;
                        } else {
                            const float cn = fmaxf(xv - a.theta, 0.f);
                            const float dd = cn - cc[h][v];
                            a.c[e] = cn;
                            a.xi[e] = fmaf(fb, dd, cn);
                            if (a.delta) a.delta[e] = dd;
                        }
                    }
                }
            }
        }
        __syncthreads();  // u is cleared for the next round
    }
}

using MarchKernel = void (*)(March);

template <int V, bool SMALL>
MarchKernel march_kernel_v(int TYT)
{
    // four depths a lane leave registers for six rows
    constexpr int most = V > 3 ? 6 : 12;
    switch (TYT) {
    case 2: return fgp_march_kernel<V, 2, SMALL>;
    case 4: return fgp_march_kernel<V, 4, SMALL>;
    case 6: return fgp_march_kernel<V, 6, SMALL>;
    case 8: return fgp_march_kernel<V, std::min(8, most), SMALL>;
    default: return fgp_march_kernel<V, most, SMALL>;
    }
}

int rows_template(int TY) { return TY <= 2 ? 2 : TY <= 4 ? 4 : TY <= 6 ? 6 : TY <= 8 ? 8 : 12; }

MarchKernel march_kernel(int V, int TY, int TX)
{
    const int r = rows_template(TY);
    const bool small = 32 * (TX + 1) <= kSmallThreads;
    switch (V) {
    case 1: return march_kernel_v<1, false>(r);
    case 2: return march_kernel_v<2, false>(r);
    case 3: return small ? march_kernel_v<3, true>(r) : march_kernel_v<3, false>(r);
    default: return small ? march_kernel_v<4, true>(r) : march_kernel_v<4, false>(r);
    }
}

size_t march_smem(int TY, int TX, int V)
{
    return ((size_t)4 * TY * TX + 3 * (TX + 1)) * 32 * V * sizeof(float);
}

}  // namespace

// Chooses the tile (h->march.TY = -1: the volume does not fit) and allocates the
// counters.  The handle's plan is set at the end, when everything it names exists: a
// call that failed leaves none.  Synchronous; not while capturing.
swopt_status march_prepare(swopt_handle* h)
{
    if (h->march.TY != 0) return SWOPT_OK;
    MarchPlan m;
    m.TY = -1;
    const int V = (h->Z + 31) / 32;
    if (V > 4) {
        h->march = m;
        return SWOPT_OK;
    }
    int sms = 0, sm_smem = 0;
    SW_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, h->device));
    SW_CUDA(cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, h->device));
    double best = 1e300;
    for (int TY = 1; TY <= std::min(h->Y, V > 3 ? 6 : 12); ++TY) {
        MarchKernel last = nullptr;
        int dmax = 0;
        cudaFuncAttributes fa;
        for (int TX = 1; TX <= std::min(h->X, 31); ++TX) {
            if (const MarchKernel k = march_kernel(V, TY, TX); k != last) {
                last = k;
                dmax = max_dynamic_smem(h, (const void*)k);
                SW_CUDA(cudaFuncGetAttributes(&fa, k));
            }
            const int threads = 32 * (TX + 1);
            const size_t smem = march_smem(TY, TX, V);
            if (threads > march_threads(rows_template(TY)) || dmax <= 0 || smem > (size_t)dmax)
                continue;
            const int regs = (fa.numRegs + 7) / 8 * 8 * 32;  // per warp
            const int warps = TX + 1;
            const int per_sm = std::min({(int)((size_t)sm_smem / (smem + 1024)), 2048 / threads,
                                         4 * (16384 / regs) / ((warps + 3) / 4 * 4), 8});
            if (per_sm < 1) continue;
            const long tiles = (long)((h->Y + TY - 1) / TY) * ((h->X + TX - 1) / TX);
            for (int SP = h->P; SP >= 1; --SP) {
                const long blocks = SP * tiles;
                if (blocks > (long)per_sm * sms) continue;
                // us per iteration of all species: the exchange, the row steps' latency and
                // their instructions (about 45 per warp and 32 depths, 2.5 per cycle)
                const double rounds = (h->P + SP - 1) / SP;
                const double busy = (double)((blocks + sms - 1) / sms);
                const double cost =
                    rounds * (1.5 + 0.1 * (TY + 1) + busy * (TY + 1) * (TX + 1) * V * 45.0 / 5000.0);
                if (cost < best) {
                    best = cost;
                    m.TY = TY;
                    m.TX = TX;
                    m.SP = SP;
                    m.blocks = (int)blocks;
                }
            }
        }
    }
    if (m.TY < 0) {
        h->march = m;
        return SWOPT_OK;
    }
    const MarchKernel k = march_kernel(V, m.TY, m.TX);
    int per_sm = 0;
    SW_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 max_dynamic_smem(h, (const void*)k)));
    SW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, 32 * (m.TX + 1),
                                                          march_smem(m.TY, m.TX, V)));
    if ((long)per_sm * sms < m.blocks) {  // the estimate was too high
        h->march = MarchPlan();
        h->march.TY = -1;
        return SWOPT_OK;
    }
    SW_CUDA(cudaMalloc((void**)&m.flags, sizeof(unsigned) * m.blocks));
    if (cudaError_t e = cudaMemset(m.flags, 0, sizeof(unsigned) * m.blocks); e != cudaSuccess) {
        cudaFree(m.flags);
        SW_CUDA(e);
    }
    h->march = m;
    return SWOPT_OK;
}

swopt_status march_launch(swopt_handle* h, const MarchCall& call, cudaStream_t st)
{
    const MarchPlan& m = h->march;
    if (m.TY <= 0 || !m.flags) {
        set_error("internal: no plan of the TV prox");
        return SWOPT_ERR_DEVICE_CHECK;
    }
    const int V = (h->Z + 31) / 32;
    March a{};
    a.z = call.z;
    a.pub[0] = h->tvr0;
    a.pub[1] = h->tvr1;
    a.P = h->P; a.Y = h->Y; a.X = h->X; a.Z = h->Z;
    a.L = nc_of(h);
    a.TY = m.TY; a.TX = m.TX;
    a.tilesY = (h->Y + m.TY - 1) / m.TY;
    a.tilesX = (h->X + m.TX - 1) / m.TX;
    a.SP = m.SP;
    a.rounds = (h->P + m.SP - 1) / m.SP;
    a.tau = call.tau;
    a.iters = call.iters;
    a.inner_momentum = call.inner_momentum;
    double t = 1.0;
    for (int i = 0; i < kMaxBetas; ++i) {
        const double t1 = 0.5 * (1.0 + std::sqrt(1.0 + 4.0 * t * t));
        a.beta[i] = call.inner_momentum == SWOPT_MOMENTUM_BECK_TEBOULLE  ? (float)((t - 1.0) / t1)
                    : call.inner_momentum == SWOPT_MOMENTUM_PAPER_PRINTED ? (float)((t - 1.0) / (t + 1.0))
                                                                          : 0.f;
        t = t1;
    }
    a.mode = call.mode;
    a.out = call.out;
    a.c = h->c;
    a.xi = h->xi;
    a.delta = call.delta;
    a.scal = h->scal;
    a.momentum = h->prm.momentum;
    a.theta = call.theta;
    a.bar = h->coop_bar;
    a.flags = m.flags;
    const MarchKernel k = march_kernel(V, m.TY, m.TX);
    SW_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 max_dynamic_smem(h, (const void*)k)));
    void* args[] = {&a};
    SW_CUDA(cudaLaunchCooperativeKernel((const void*)k, dim3(m.blocks), dim3(32 * (m.TX + 1)), args,
                                        march_smem(m.TY, m.TX, V), st));
    SW_LAUNCHED(h);
    return SWOPT_OK;
}

}  // namespace swopt
