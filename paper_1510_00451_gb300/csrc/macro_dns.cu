// Macro solver for Eq. (homo) and direct simulation of Eq. (model).
//
// Macro step (HMM step 4): U_t = div(K grad U) in conservative flux form on
// the periodic N x N grid, face tensors K_f = (K_node + K_neighbour)/2, the
// mixed term by the 4-point average of cross differences (9-point stencil),
// Heun's RK2.  Every face flux is evaluated by both adjacent cells with the
// same operations, so sum(U) telescopes exactly apart from summation rounding.
// Small grids: one CTA keeps U and U* in shared memory and its face coefficients in
// registers for all steps.  Larger ones: tiles, each CTA taking a tile with a halo
// through several steps per launch (the halo's outer rings are recomputed).
// The mass H^2 sum(U) of every step is summed in FP64.
//
// DNS: u_t = v1 D0x u + v2 D0y u + kappa (Dxx + Dyy) u, v = (-D0y psi, D0x psi),
// both RK stages fused per tile.  Large periodic grids: u and psi staged with a halo of 2
// in shared memory, one pass over HBM per time step (read u, read psi, write u).  Grids up to
// 1024^2, and Dirichlet in x1 in FP32: four steps of a tile with its halo per launch.  Dirichlet in
// FP64: a step per launch, from coefficients formed once per run.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <mutex>
#include <string>
#include <vector>

#include <cuda.h>

#include "async_copy.cuh"
#include "mlsd_internal.cuh"

namespace mlsd {
namespace {

// deterministic FP64 block sum (all threads return the total)
__device__ double block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
}

// Face coefficients of the flux form, scaled by dt / H: with the face tensors
// K_f = (K_node + K_neighbour) / 2, the east face (i+1/2, j) of cell (i, j) carries
//   fe = aE (uE - u) + cE (Dc + DE),   aE = dt K11_f / H^2, cE = dt K12_f / (4 H^2),
// D = u(j+1) - u(j-1) of a column, the north face (i, j+1/2)
//   fn = aN (uN - u) + cN (Gc + GN),   aN = dt K22_f / H^2, cN = dt K12_f / (4 H^2),
// G = u(i+1) - u(i-1) of a row, and dt div(K grad U) = (fe - fw) + (fn - fs), the west and
// south fluxes being the neighbours' east and north ones formed from the same operands.
// Coefficient q (0: aE, 1: cE, 2: aN, 3: cN) of cell (i, j) from the node tensors; f = dt / (2 H^2)
template <typename real>
__device__ __forceinline__ real macro_face(int q, const double *Kg, int N, int i, int j, real f)
{
    const int c = j * N + i;
    const int o = q < 2 ? j * N + (i + 1 == N ? 0 : i + 1) : (j + 1 == N ? 0 : j + 1) * N + i;
    const int k = q == 0 ? 0 : (q == 2 ? 2 : 1);
    return ((q & 1) ? (real)0.25 * f : f) * ((real)Kg[3LL * c + k] + (real)Kg[3LL * o + k]);
}

// coefficients into co [4][N][N] (above 23170^2 cells they do not fit 32-bit indices); U into V when
// V is given; with dir, column 0 of U (and V) takes the boundary value ul
template <typename real>
__global__ void k_macro_prep(int N, const double *Kg, real f, real *co, real *U, real *V, int dir,
                             real ul)
{
    const int c = blockIdx.x * blockDim.x + threadIdx.x, NN = N * N;
    if (c >= NN) return;
    const int i = c % N, j = c / N;
#pragma unroll
    for (int q = 0; q < 4; ++q) co[(long long)q * NN + c] = macro_face(q, Kg, N, i, j, f);
    if (dir && i == 0) U[c] = ul;
    if (V) V[c] = (dir && i == 0) ? ul : U[c];
}

// The R cells (x, y0 .. y0+R-1) of a thread: their coefficients, and one Heun stage.
template <typename real, int R>
struct MacroStrip {
    real aE[R], cE[R], aW[R], cW[R], aN[R + 1], cN[R + 1];   // aN[r]: south face of row r

    // coefficients co(q, i, j) of the cells at columns gx (west neighbour gw) and rows gy(r),
    // r = -1 .. R-1
    template <typename Co, typename Row>
    __device__ __forceinline__ void load(Co co, int gx, int gw, Row gy)
    {
#pragma unroll
        for (int r = 0; r <= R; ++r) {
            const int j = gy(r - 1);
            aN[r] = co(2, gx, j);
            cN[r] = co(3, gx, j);
            if (r > 0) {
                aE[r - 1] = co(0, gx, j); cE[r - 1] = co(1, gx, j);
                aW[r - 1] = co(0, gw, j); cW[r - 1] = co(1, gw, j);
            }
        }
    }

    // out[r] = dt div(K grad X) of the strip's cells; X(row r = -1 .. R, column -1 | 0 | 1)
    template <typename Get>
    __device__ __forceinline__ void rhs(Get X, real (&out)[R]) const
    {
        real wm = X(-1, -1), cm = X(-1, 0), em = X(-1, 1);
        real w = X(0, -1), c = X(0, 0), e = X(0, 1);
        real g = e - w;
        // south flux of row 0
        real fs = fma(aN[0], c - cm, cN[0] * (g + (em - wm)));
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const real wp = X(r + 1, -1), cp = X(r + 1, 0), ep = X(r + 1, 1);
            const real Dw = wp - wm, Dc = cp - cm, De = ep - em, gp = ep - wp;
            const real fe = fma(aE[r], e - c, cE[r] * (Dc + De));
            const real fw = fma(aW[r], c - w, cW[r] * (Dc + Dw));
            const real fn = fma(aN[r + 1], cp - c, cN[r + 1] * (g + gp));
            out[r] = (fe - fw) + (fn - fs);
            fs = fn;
            wm = w; cm = c; em = e;
            w = wp; c = cp; e = ep;
            g = gp;
        }
    }
};

// One CTA, the whole grid in shared memory for all steps, a thread a cell with its eight face
// coefficients in registers.  DIR: the Sec. 4 set-up, Dirichlet in x1 -- column 0 is the
// boundary x1 = 0 (held) and the virtual column N the boundary x1 = 2 pi with value ur; the K
// field stays periodic.
template <typename real, int NT, bool DIR>
__global__ void __launch_bounds__(NT) k_macro_resident(int N, real *Ug, const double *Kg, real f,
                                                       int nsteps, double *mass, real ul, real ur)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    real *U = reinterpret_cast<real *>(smem_raw), *Us = U + N * N;
    __shared__ double red[32];
    const int c = threadIdx.x, x = c % N, y = c / N;
    const bool own = y < N;
    const double H = 2.0 * kPi / N, H2 = H * H;
    const int xe = x + 1 == N ? 0 : x + 1, xw = x == 0 ? N - 1 : x - 1;
    const int yn = y + 1 >= N ? 0 : y + 1, ys = y == 0 ? N - 1 : y - 1;
    const bool held = DIR && x == 0, east = DIR && x + 1 == N;
    MacroStrip<real, 1> st;
    real u = 0, d[1], s;
    double m = 0.0;
    if (own) {
        st.load([&](int q, int i, int j) { return macro_face(q, Kg, N, i, j, f); }, x, xw,
                [&](int r) { return r < 0 ? ys : y; });
        u = held ? ul : Ug[c];
        U[c] = u;
        m = (double)u;
    }
    m = block_sum(m, red);
    if (threadIdx.x == 0 && mass) mass[0] = m * H2;
    const int row[3] = {ys * N, y * N, yn * N};
    auto stage = [&](const real *X) {
        st.rhs([&](int r, int k) {
            return k == 0 ? X[row[r + 1] + x] : k < 0 ? X[row[r + 1] + xw] : (east ? ur : X[row[r + 1] + xe]);
        }, d);
    };
    for (int k = 0; k < nsteps; ++k) {
        if (own) {
            stage(U);
            s = held ? u : u + d[0];
            Us[c] = s;
        }
        __syncthreads();
        m = 0.0;
        if (own) {
            stage(Us);
            u = held ? u : (real)0.5 * (u + s + d[0]);
            U[c] = u;
            m = (double)u;
        }
        if (mass) {
            m = block_sum(m, red);
            if (threadIdx.x == 0) mass[k + 1LL] = m * H2;
        }
        __syncthreads();
    }
    if (own) Ug[c] = u;
}

// `steps` <= S Heun steps of one TX x TY tile per CTA.  The tile comes with a halo of 2 S
// cells; each stage is valid on one ring less, so strips of R rows outside a stage's valid
// rows are skipped, the rest of the rim is computed with clamped neighbours and never
// stored.  What bounds it: latency (a launch, two barriers a step), in FP64 issue beside it.
// A step at 128^2: FP32 1.14 us, against 10.0 with a launch per Heun stage that formed every
// face from K again, 1.54 without overlapping the launches; FP64 5.2 us against 16.6.
// With part, the tile's share of sum(U) after step k goes to
// part[k * tiles + tile].
template <typename real, int TX, int TY, int S, bool DIR>
struct MacroTile {
    static constexpr int HALO = 2 * S, EX = TX + 2 * HALO, EY = TY + 2 * HALO;
    static constexpr int R = sizeof(real) == 8 ? 1 : 4;
    static constexpr int NT = EX * EY / R;
    static_assert(EY % R == 0 && NT <= 1024, "strips of R rows");
};
template <typename real, int TX, int TY, int S, bool DIR>
__global__ void __launch_bounds__((MacroTile<real, TX, TY, S, DIR>::NT + 31) / 32 * 32)
k_macro_tile(int N, const real *Uin, real *Uout, const real *__restrict__ co,
             int steps, double *part, real ur)
{
    using M = MacroTile<real, TX, TY, S, DIR>;
    constexpr int EX = M::EX, EY = M::EY, R = M::R, HALO = M::HALO;
    __shared__ real U[EY * EX], Us[EY * EX];
    __shared__ double red[32];
    const int t = threadIdx.x, x = t % EX, y0 = t / EX * R;
    const bool own = t < M::NT;                     // the last warp may be partial
    const int gx0 = blockIdx.x * TX - HALO + x;     // grid column before the periodic wrap
    const int gx = ((gx0 % N) + N) % N, gw = gx == 0 ? N - 1 : gx - 1;
    auto gy = [&](int r) { const int y = (int)blockIdx.y * TY - HALO + y0 + r; return ((y % N) + N) % N; };
    const bool held = DIR && (gx0 == 0 || gx0 == N);
    MacroStrip<real, R> st;
    real u[R], d[R], s[R];
    if (own) st.load([&](int q, int i, int j) { return co[((long long)q * N + j) * N + i]; }, gx, gw, gy);
    chain_wait();
    if (own) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            u[r] = (DIR && gx0 == N) ? ur : Uin[(long long)gy(r) * N + gx];
            U[(y0 + r) * EX + x] = u[r];
        }
    }
    // cells of the tile that are inside the grid
    const bool colin = own && x >= HALO && x < HALO + TX && gx0 < N;
    auto inside = [&](int r) {
        return colin && y0 + r >= HALO && y0 + r < HALO + TY && (int)blockIdx.y * TY - HALO + y0 + r < N;
    };
    __syncthreads();
    const int xw = x > 0 ? -1 : 0, xe = x < EX - 1 ? 1 : 0;
    const int ym = y0 > 0 ? y0 - 1 : 0, yp = y0 + R < EY ? y0 + R : EY - 1;
    auto stage = [&](const real *X) {
        st.rhs([&](int r, int k) {
            return X[(r < 0 ? ym : r == R ? yp : y0 + r) * EX + x + (k < 0 ? xw : k > 0 ? xe : 0)];
        }, d);
    };
    for (int k = 0; k < steps; ++k) {
        if (own && y0 + R > 2 * k + 1 && y0 < EY - 1 - 2 * k) {
            stage(U);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                s[r] = held ? u[r] : u[r] + d[r];
                Us[(y0 + r) * EX + x] = s[r];
            }
        }
        __syncthreads();
        double m = 0.0;
        if (own && y0 + R > 2 * k + 2 && y0 < EY - 2 - 2 * k) {
            stage(Us);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                u[r] = held ? u[r] : (real)0.5 * (u[r] + s[r] + d[r]);
                U[(y0 + r) * EX + x] = u[r];
                if (part && inside(r)) m += (double)u[r];
            }
        }
        if (part) {
            m = block_sum(m, red);
            if (t == 0)
                part[(long long)k * gridDim.x * gridDim.y + blockIdx.y * gridDim.x + blockIdx.x] = m;
        }
        __syncthreads();
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
        if (inside(r)) Uout[(long long)gy(r) * N + gx] = u[r];
}

// Dirichlet set-up: column 0 (the boundary x1 = 0) takes the boundary value
template <typename real>
__global__ void k_set_col0(int N, real *U, real ul)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j < N) U[(long long)j * N] = ul;
}

template <typename real>
__global__ void k_mass_part(int NN, const real *U, double *part)
{
    __shared__ double red[32];
    const int c = blockIdx.x * blockDim.x + threadIdx.x;
    double m = c < NN ? (double)U[c] : 0.0;
    m = block_sum(m, red);
    if (threadIdx.x == 0) part[blockIdx.x] = m;
}

// mass[s] = H^2 * sum_b part[s][b]
__global__ void k_mass_final(int nsteps1, int nblocks, const double *part, double H2, double *mass)
{
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= nsteps1) return;
    double t = 0.0;
    for (int b = 0; b < nblocks; ++b) t += part[(long long)s * nblocks + b];
    mass[s] = t * H2;
}

__global__ void k_kmax(int NN, const double *K, double *out)
{
    __shared__ double red[32];
    double m = 0.0;
    for (int c = threadIdx.x; c < NN; c += blockDim.x)
        m = fmax(m, K[3 * c] + K[3 * c + 2] + fabs(K[3 * c + 1]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, red[w]);
        *out = t;
    }
}

// ---------------------------------------------------------------------------
// DNS step, both Heun stages fused, one pass over HBM (read u, read psi,
// write u).  A CTA owns a 128 x 64 output tile.  u and psi are staged with a
// 2-row / 8-column halo by 16-byte cp.async copies.  Thread (g, seg) owns the
// 4 columns x0 - 4 + 4g .. +3 (g = 0 and 33 are halo groups) and the 8 output
// rows y0 + 8 seg .. +7: it computes stage 1 on those rows plus one row above
// and below (kept in registers), publishes its left and right edge columns of
// the stage-1 field for its own rows, and after one barrier computes stage 2
// on its output rows from registers (north, south) and the neighbours' edges
// (east, west).
constexpr int DTX = 128, DRS = 8;
constexpr int DG = DTX / 4 + 2;                // column groups incl. the two halo groups
constexpr int DLX = DTX + 16;                  // staged columns x0-8 .. x0+TX+7
template <int DTY> struct DnsTile {
    static constexpr int DSEG = DTY / DRS;     // row segments
    static constexpr int DTH = DG * DSEG;      // threads
    static constexpr int DLY = DTY + 4;        // staged rows y0-2 .. y0+TY+1
    static constexpr size_t SMEM = (size_t)2 * DLY * DLX * 4 + (size_t)2 * DTY * DG * 4;
};

__device__ __forceinline__ void cp16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::
                 "r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}

// Both Heun stages of one tile from its staged u and psi (rows y0-2 .. y0+DTY+1,
// columns x0-8 .. x0+DTX+7 in su, sp): stage 1 in registers, the edge columns
// of the stage-1 field through eL / eR and one CTA barrier, stage 2 stored to un.
template <int DTY>
__device__ __forceinline__ void dns_tile(const float *su, const float *sp, float *eL, float *eR,
                                         int nf, int x0, int y0, float *__restrict__ un, float ax,
                                         float kd, float dt)
{
    constexpr int DTH = DnsTile<DTY>::DTH;
    const int g = threadIdx.x % DG, seg = threadIdx.x / DG;
    const int c0 = 4 + 4 * g;                 // staged column of the group's first column
    // the last warp is partial (DTH = 34 DTY/8 threads): shuffles name its lanes only;
    // its last thread is a g = DG - 1 thread, so no lane reads past it
    const int lane = threadIdx.x & 31, wbase = threadIdx.x & ~31;
    const unsigned wmask = DTH - wbase >= 32 ? 0xffffffffu : ((1u << (DTH - wbase)) - 1u);
    const bool edgeW = g == 0 || lane == 0, edgeE = g == DG - 1 || lane == 31;
    // x + dt f(x) = x + cD (xE + xW + xN + xS - 4 x)
    //                 + cA [(psiS - psiN)(xE - xW) + (psiE - psiW)(xN - xS)],
    // cA = dt / (4 h^2), cD = dt kappa / h^2; the Laplacian stays a difference so
    // that rounding does not bias the sum of u
    const float cA = dt * ax * ax, cD = dt * kd;
    const int rbase = 2 + DRS * seg;          // staged row of the segment's first output row
    // ---- stage 1 on rows rbase-1 .. rbase+DRS (registers s[0..DRS+1]) ----
    float s1[DRS + 2][4];
    {
        float um[4], uc[4], up[4], pm[4], pc[4], pp[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            um[c] = su[(rbase - 2) * DLX + c0 + c]; uc[c] = su[(rbase - 1) * DLX + c0 + c];
            pm[c] = sp[(rbase - 2) * DLX + c0 + c]; pc[c] = sp[(rbase - 1) * DLX + c0 + c];
        }
#pragma unroll
        for (int k = 0; k < DRS + 2; ++k) {
            const int r = rbase - 1 + k;
            const float4 un4 = *reinterpret_cast<const float4 *>(su + (r + 1) * DLX + c0);
            const float4 pn4 = *reinterpret_cast<const float4 *>(sp + (r + 1) * DLX + c0);
            up[0] = un4.x; up[1] = un4.y; up[2] = un4.z; up[3] = un4.w;
            pp[0] = pn4.x; pp[1] = pn4.y; pp[2] = pn4.z; pp[3] = pn4.w;
            // the neighbouring columns come from the neighbouring lanes (the groups of a
            // segment are consecutive threads); lanes at a warp or segment edge read
            // shared memory (a scalar column read is a 4-way bank conflict)
            float uw = __shfl_up_sync(wmask, uc[3], 1), ue = __shfl_down_sync(wmask, uc[0], 1);
            float pw = __shfl_up_sync(wmask, pc[3], 1), pe = __shfl_down_sync(wmask, pc[0], 1);
            if (edgeW) { uw = su[r * DLX + c0 - 1]; pw = sp[r * DLX + c0 - 1]; }
            if (edgeE) { ue = su[r * DLX + c0 + 4]; pe = sp[r * DLX + c0 + 4]; }
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float uE = c < 3 ? uc[c + 1] : ue, uW = c > 0 ? uc[c - 1] : uw;
                const float pE = c < 3 ? pc[c + 1] : pe, pW = c > 0 ? pc[c - 1] : pw;
                float t = (pm[c] - pp[c]) * (uE - uW);
                t = fmaf(pE - pW, up[c] - um[c], t);
                const float lap = fmaf(-4.0f, uc[c], (uE + uW) + (up[c] + um[c]));
                s1[k][c] = fmaf(cA, t, fmaf(cD, lap, uc[c]));
            }
#pragma unroll
            for (int c = 0; c < 4; ++c) { um[c] = uc[c]; uc[c] = up[c]; pm[c] = pc[c]; pc[c] = pp[c]; }
        }
    }
    // publish the edge columns of the stage-1 field on the segment's own rows
#pragma unroll
    for (int k = 0; k < DRS; ++k) {
        eL[(DRS * seg + k) * DG + g] = s1[k + 1][0];
        eR[(DRS * seg + k) * DG + g] = s1[k + 1][3];
    }
    __syncthreads();
    // ---- stage 2 on the output rows (the halo groups hold stage-1 values only) ----
    if (g != 0 && g != DG - 1) {
        float pm[4], pc[4], pp[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            pm[c] = sp[(rbase - 1) * DLX + c0 + c];
            pc[c] = sp[rbase * DLX + c0 + c];
        }
        const int gx = x0 + 4 * (g - 1);
#pragma unroll
        for (int k = 0; k < DRS; ++k) {
            const int r = rbase + k;
            const float4 pn4 = *reinterpret_cast<const float4 *>(sp + (r + 1) * DLX + c0);
            pp[0] = pn4.x; pp[1] = pn4.y; pp[2] = pn4.z; pp[3] = pn4.w;
            const float pw = sp[r * DLX + c0 - 1], pe = sp[r * DLX + c0 + 4];
            const float sw = eR[(DRS * seg + k) * DG + g - 1], se = eL[(DRS * seg + k) * DG + g + 1];
            const float4 u4 = *reinterpret_cast<const float4 *>(su + r * DLX + c0);
            const float uo[4] = {u4.x, u4.y, u4.z, u4.w};
            float o[4];
            // (u + s + dt f(s)) / 2
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                const float sC = s1[k + 1][c], sN = s1[k + 2][c], sS = s1[k][c];
                const float sE = c < 3 ? s1[k + 1][c + 1] : se, sW = c > 0 ? s1[k + 1][c - 1] : sw;
                const float pE = c < 3 ? pc[c + 1] : pe, pW = c > 0 ? pc[c - 1] : pw;
                float t = (pm[c] - pp[c]) * (sE - sW);
                t = fmaf(pE - pW, sN - sS, t);
                const float lap = fmaf(-4.0f, sC, (sE + sW) + (sN + sS));
                o[c] = 0.5f * (uo[c] + fmaf(cA, t, fmaf(cD, lap, sC)));
            }
            *reinterpret_cast<float4 *>(un + (long long)(y0 + DRS * seg + k) * nf + gx) =
                make_float4(o[0], o[1], o[2], o[3]);
#pragma unroll
            for (int c = 0; c < 4; ++c) { pm[c] = pc[c]; pc[c] = pp[c]; }
        }
    }
}

// f32x2 helpers: a - b as fma(b, -1, a), which rounds like the subtraction
__device__ __forceinline__ float2 sub2(float2 a, float2 b)
{
    return __ffma2_rn(b, make_float2(-1.f, -1.f), a);
}
__device__ __forceinline__ float2 bcast2(float v) { return make_float2(v, v); }

// dns_tile with the columns of a thread's group in f32x2 pairs (0, 1) and (2, 3):
// every stencil operation is one FFMA2 / FADD2 / FMUL2 for two cells, with the
// same operands and order per cell as dns_tile, so the result is the same bit
// for bit.  The neighbour pairs that straddle the two halves, (1, 2), (w, 0) and
// (3, e), are assembled from registers.
template <int DTY>
__device__ __forceinline__ void dns_tile2(const float *su, const float *sp, float *eL, float *eR,
                                          int nf, int x0, int y0, float *__restrict__ un, float ax,
                                          float kd, float dt)
{
    constexpr int DTH = DnsTile<DTY>::DTH;
    const int g = threadIdx.x % DG, seg = threadIdx.x / DG;
    const int c0 = 4 + 4 * g;
    const int lane = threadIdx.x & 31, wbase = threadIdx.x & ~31;
    const unsigned wmask = DTH - wbase >= 32 ? 0xffffffffu : ((1u << (DTH - wbase)) - 1u);
    const bool edgeW = g == 0 || lane == 0, edgeE = g == DG - 1 || lane == 31;
    const float2 cA = bcast2(dt * ax * ax), cD = bcast2(dt * kd), m4 = bcast2(-4.0f);
    const int rbase = 2 + DRS * seg;
    float2 sA[DRS + 2], sB[DRS + 2];             // stage-1 field, columns (0, 1) and (2, 3)
    {
        auto ld2 = [&](const float *base, int r, float2 &a, float2 &b) {
            const float4 v = *reinterpret_cast<const float4 *>(base + r * DLX + c0);
            a = make_float2(v.x, v.y);
            b = make_float2(v.z, v.w);
        };
        float2 umA, umB, ucA, ucB, pmA, pmB, pcA, pcB;
        ld2(su, rbase - 2, umA, umB); ld2(su, rbase - 1, ucA, ucB);
        ld2(sp, rbase - 2, pmA, pmB); ld2(sp, rbase - 1, pcA, pcB);
#pragma unroll
        for (int k = 0; k < DRS + 2; ++k) {
            const int r = rbase - 1 + k;
            float2 upA, upB, ppA, ppB;
            ld2(su, r + 1, upA, upB);
            ld2(sp, r + 1, ppA, ppB);
            float uw = __shfl_up_sync(wmask, ucB.y, 1), ue = __shfl_down_sync(wmask, ucA.x, 1);
            float pw = __shfl_up_sync(wmask, pcB.y, 1), pe = __shfl_down_sync(wmask, pcA.x, 1);
            if (edgeW) { uw = su[r * DLX + c0 - 1]; pw = sp[r * DLX + c0 - 1]; }
            if (edgeE) { ue = su[r * DLX + c0 + 4]; pe = sp[r * DLX + c0 + 4]; }
            const float2 uMid = make_float2(ucA.y, ucB.x), pMid = make_float2(pcA.y, pcB.x);
            const float2 uWA = make_float2(uw, ucA.x), uEB = make_float2(ucB.y, ue);
            const float2 pWA = make_float2(pw, pcA.x), pEB = make_float2(pcB.y, pe);
            {   // columns 0, 1: east (1, 2), west (w, 0)
                float2 t = __fmul2_rn(sub2(pmA, ppA), sub2(uMid, uWA));
                t = __ffma2_rn(sub2(pMid, pWA), sub2(upA, umA), t);
                const float2 lap = __ffma2_rn(m4, ucA, __fadd2_rn(__fadd2_rn(uMid, uWA),
                                                                 __fadd2_rn(upA, umA)));
                sA[k] = __ffma2_rn(cA, t, __ffma2_rn(cD, lap, ucA));
            }
            {   // columns 2, 3: east (3, e), west (1, 2)
                float2 t = __fmul2_rn(sub2(pmB, ppB), sub2(uEB, uMid));
                t = __ffma2_rn(sub2(pEB, pMid), sub2(upB, umB), t);
                const float2 lap = __ffma2_rn(m4, ucB, __fadd2_rn(__fadd2_rn(uEB, uMid),
                                                                 __fadd2_rn(upB, umB)));
                sB[k] = __ffma2_rn(cA, t, __ffma2_rn(cD, lap, ucB));
            }
            umA = ucA; umB = ucB; ucA = upA; ucB = upB;
            pmA = pcA; pmB = pcB; pcA = ppA; pcB = ppB;
        }
    }
#pragma unroll
    for (int k = 0; k < DRS; ++k) {
        eL[(DRS * seg + k) * DG + g] = sA[k + 1].x;
        eR[(DRS * seg + k) * DG + g] = sB[k + 1].y;
    }
    __syncthreads();
    if (g != 0 && g != DG - 1) {
        const float4 pm4 = *reinterpret_cast<const float4 *>(sp + (rbase - 1) * DLX + c0);
        const float4 pc4 = *reinterpret_cast<const float4 *>(sp + rbase * DLX + c0);
        float2 pmA = make_float2(pm4.x, pm4.y), pmB = make_float2(pm4.z, pm4.w);
        float2 pcA = make_float2(pc4.x, pc4.y), pcB = make_float2(pc4.z, pc4.w);
        const int gx = x0 + 4 * (g - 1);
        const float2 half = bcast2(0.5f);
#pragma unroll
        for (int k = 0; k < DRS; ++k) {
            const int r = rbase + k;
            const float4 pn4 = *reinterpret_cast<const float4 *>(sp + (r + 1) * DLX + c0);
            const float2 ppA = make_float2(pn4.x, pn4.y), ppB = make_float2(pn4.z, pn4.w);
            const float pw = sp[r * DLX + c0 - 1], pe = sp[r * DLX + c0 + 4];
            const float sw = eR[(DRS * seg + k) * DG + g - 1], se = eL[(DRS * seg + k) * DG + g + 1];
            const float4 u4 = *reinterpret_cast<const float4 *>(su + r * DLX + c0);
            const float2 uoA = make_float2(u4.x, u4.y), uoB = make_float2(u4.z, u4.w);
            const float2 sCA = sA[k + 1], sCB = sB[k + 1];
            const float2 sMid = make_float2(sCA.y, sCB.x), pMid = make_float2(pcA.y, pcB.x);
            const float2 sWA = make_float2(sw, sCA.x), sEB = make_float2(sCB.y, se);
            const float2 pWA = make_float2(pw, pcA.x), pEB = make_float2(pcB.y, pe);
            float2 oA, oB;
            {
                float2 t = __fmul2_rn(sub2(pmA, ppA), sub2(sMid, sWA));
                t = __ffma2_rn(sub2(pMid, pWA), sub2(sA[k + 2], sA[k]), t);
                const float2 lap = __ffma2_rn(m4, sCA, __fadd2_rn(__fadd2_rn(sMid, sWA),
                                                                 __fadd2_rn(sA[k + 2], sA[k])));
                oA = __fmul2_rn(half, __fadd2_rn(uoA, __ffma2_rn(cA, t, __ffma2_rn(cD, lap, sCA))));
            }
            {
                float2 t = __fmul2_rn(sub2(pmB, ppB), sub2(sEB, sMid));
                t = __ffma2_rn(sub2(pEB, pMid), sub2(sB[k + 2], sB[k]), t);
                const float2 lap = __ffma2_rn(m4, sCB, __fadd2_rn(__fadd2_rn(sEB, sMid),
                                                                 __fadd2_rn(sB[k + 2], sB[k])));
                oB = __fmul2_rn(half, __fadd2_rn(uoB, __ffma2_rn(cA, t, __ffma2_rn(cD, lap, sCB))));
            }
            *reinterpret_cast<float4 *>(un + (long long)(y0 + DRS * seg + k) * nf + gx) =
                make_float4(oA.x, oA.y, oB.x, oB.y);
            pmA = pcA; pmB = pcB; pcA = ppA; pcB = ppB;
        }
    }
}

template <int DTY>
__global__ void __launch_bounds__(DnsTile<DTY>::DTH) k_dns_step(int nf, const float *u,
                                                               const float *__restrict__ psi,
                                                               float *un, float ax, float kd, float dt)
{
    constexpr int DLY = DnsTile<DTY>::DLY, DTH = DnsTile<DTY>::DTH;
    extern __shared__ __align__(16) float dsm[];
    float *su = dsm;                          // [DLY][DLX]
    float *sp = su + DLY * DLX;               // [DLY][DLX]
    float *eL = sp + DLY * DLX;               // [DTY][DG]  stage-1 value of a group's column 0
    float *eR = eL + DTY * DG;                // [DTY][DG]  ... of its column 3
    const int x0 = blockIdx.x * DTX, y0 = blockIdx.y * DTY;
    chain_wait();
    for (int k = threadIdx.x; k < DLY * (DLX / 4); k += DTH) {
        const int r = k / (DLX / 4), q = k % (DLX / 4);
        int gy = y0 - 2 + r; gy = gy < 0 ? gy + nf : (gy >= nf ? gy - nf : gy);
        int gx = x0 - 8 + 4 * q; gx = gx < 0 ? gx + nf : (gx >= nf ? gx - nf : gx);
        const long long off = (long long)gy * nf + gx;
        cp16(su + r * DLX + 4 * q, u + off);
        cp16(sp + r * DLX + 4 * q, psi + off);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    dns_tile<DTY>(su, sp, eL, eR, nf, x0, y0, un, ax, kd, dt);
}

// Persistent variant: each CTA takes tiles from a queue (an atomic counter per
// launch; two counters alternate, and each launch zeroes the next one's) into
// NBUF staging buffers.  Thread 0 loads a tile's u and psi boxes by two 2-D
// tensor copies (one box of DLX x DLY each, starting at (x0 - 8, y0 - 2)) that
// complete on the buffer's mbarrier; the buffer's next tile is claimed and its
// copy issued as soon as the buffer is free, so with NBUF = 2 it lands while
// this CTA computes the other buffer's tile.
// A launch of a run starts while its predecessor ends (8192^2: 146.7 -> 144.3 us a
// step, 2048^2: 18.0 -> 15.5, of which the tail of a launch is the most).
// Boxes reaching past the grid's edge are zero-filled by the copy; the threads
// then put in the periodic images from global memory.  A wait that runs out
// (about a second) latches MLSD_ETIMEOUT into g_dns_status and ends the CTA's
// walk after a second bounded wait for each copy it has issued.
__device__ int g_dns_status;

template <int DTY, int NBUF>
struct DnsTma {
    static constexpr int DLY = DnsTile<DTY>::DLY;
    static constexpr int FIELD = DLY * DLX;                        // floats per staged field
    static constexpr int BUF = (2 * FIELD * 4 + 1023) / 1024 * 256; // floats per buffer (1 KB steps)
    static constexpr size_t SMEM = 1024 + (size_t)NBUF * BUF * 4 + (size_t)2 * DTY * DG * 4;
    static constexpr uint32_t BYTES = 2u * FIELD * 4u;              // one tile's copies
};

template <int DTY, int NBUF, bool PAIR>
__global__ void __launch_bounds__(DnsTile<DTY>::DTH)
k_dns_tma(const __grid_constant__ CUtensorMap mu, const __grid_constant__ CUtensorMap mp, int nf,
          const float *u, const float *__restrict__ psi, float *un,
          float ax, float kd, float dt, int *queue, int which)
{
    using T = DnsTma<DTY, NBUF>;
    constexpr int DLY = T::DLY, DTH = DnsTile<DTY>::DTH;
    extern __shared__ __align__(16) unsigned char dsm_raw[];
    __shared__ __align__(8) uint64_t full[NBUF];
    __shared__ int tile_of[NBUF];
    // the copies land at 1 KB-aligned buffers
    float *base = reinterpret_cast<float *>(dsm_raw + ((1024 - (smem_addr(dsm_raw) & 1023)) & 1023));
    float *eL = base + NBUF * T::BUF, *eR = eL + DTY * DG;
    const int tiles_x = nf / DTX, ntiles = tiles_x * (nf / DTY);
    const CUtensorMap *pmu = &mu, *pmp = &mp;
    // claim the next tile of the launch for buffer b and start its copies; past the
    // last tile, a plain arrival completes the phase so that the CTA's wait ends
    auto claim = [&](int b) {
        const int t = atomicAdd(&queue[which], 1);
        tile_of[b] = t;
        const uint32_t mb = smem_addr(&full[b]);
        if (t < ntiles) {
            const int x0 = (t % tiles_x) * DTX, y0 = (t / tiles_x) * DTY;
            float *su = base + b * T::BUF;
            mbar_expect(mb, T::BYTES);
            tma_load_2d(smem_addr(su), pmu, x0 - 8, y0 - 2, mb);
            tma_load_2d(smem_addr(su + T::FIELD), pmp, x0 - 8, y0 - 2, mb);
        } else {
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" :: "r"(mb) : "memory");
        }
    };
    if (threadIdx.x == 0) {
        for (int b = 0; b < NBUF; ++b) mbar_init1(smem_addr(&full[b]));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    chain_wait();
    if (threadIdx.x == 0) {
        if (blockIdx.x == 0) queue[which ^ 1] = 0;      // the next launch's queue
        for (int b = 0; b < NBUF; ++b) claim(b);
    }
    __syncthreads();                                     // the mbarriers are initialised
    for (int k = 0;; ++k) {
        const int b = k % NBUF;
        const uint32_t mb = smem_addr(&full[b]), par = (uint32_t)((k / NBUF) & 1);
        const bool ok = mbar_wait_bounded(mb, par);
        if (__syncthreads_or(!ok)) {
            if (threadIdx.x == 0) {
                atomicCAS(&g_dns_status, 0, MLSD_ETIMEOUT);
                // the copies of this and the other buffers, if still coming
                for (int j = 0; j < NBUF; ++j)
                    if (tile_of[(k + j) % NBUF] < ntiles)
                        mbar_wait_bounded(smem_addr(&full[(k + j) % NBUF]),
                                          (uint32_t)(((k + j) / NBUF) & 1));
            }
            break;
        }
        const int t = tile_of[b];
        if (t >= ntiles) break;                         // claims only grow: no copy is pending
        const int x0 = (t % tiles_x) * DTX, y0 = (t / tiles_x) * DTY;
        float *su = base + b * T::BUF, *sp = su + T::FIELD;
        if (x0 == 0 || x0 + DTX == nf || y0 == 0 || y0 + DTY == nf) {
            // periodic images of the staged cells outside the grid
            for (int e = threadIdx.x; e < DLY * DLX; e += DTH) {
                const int r = e / DLX, c = e % DLX;
                int gy = y0 - 2 + r, gx = x0 - 8 + c;
                if (gy >= 0 && gy < nf && gx >= 0 && gx < nf) continue;
                gy = gy < 0 ? gy + nf : (gy >= nf ? gy - nf : gy);
                gx = gx < 0 ? gx + nf : (gx >= nf ? gx - nf : gx);
                su[e] = __ldcg(u + (long long)gy * nf + gx);   // written by the launch before
                sp[e] = psi[(long long)gy * nf + gx];
            }
            __syncthreads();
        }
        if constexpr (PAIR) dns_tile2<DTY>(su, sp, eL, eR, nf, x0, y0, un, ax, kd, dt);
        else dns_tile<DTY>(su, sp, eL, eR, nf, x0, y0, un, ax, kd, dt);
        // every thread's reads and writes of this buffer come before the next copy into it
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (threadIdx.x == 0) claim(b);
    }
}

// Failure-path check of the tile wait: one thread waits on a fresh mbarrier that
// receives no arrival and no copy, so the wait runs out and latches MLSD_ETIMEOUT
__global__ void k_wait_check_tile(int *status)
{
    __shared__ __align__(8) uint64_t mb;
    if (threadIdx.x == 0) {
        mbar_init1(smem_addr(&mb));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        if (!mbar_wait_bounded(smem_addr(&mb), 0)) atomicCAS(status, 0, MLSD_ETIMEOUT);
    }
}

// Several Heun steps of one tile per CTA (FP32): grids that the chip's L2 holds, where a
// launch per step is mostly latency.  The tile comes with a halo of 2 S cells and the whole
// run of `steps` <= S steps stays on chip; each stage is valid on one ring less, so strips
// outside a stage's valid rows are skipped and the rest of the rim is computed with clamped
// neighbours and never stored.  A thread owns R rows of one column: its cells and the psi
// differences that multiply them live in registers, the field goes through shared memory
// once per stage.  The arithmetic per cell is dns_tile's, operand for operand:
//   x + dt f(x) = x + cD (xE + xW + xN + xS - 4 x)
//                   + cA [(psiS - psiN)(xE - xW) + (psiE - psiW)(xN - xS)].
// DIR: Dirichlet in x1 (column 0 held at ul, the virtual column nf at ur), periodic in x2;
// psi and the velocity stay periodic.  What bounds it: at 512^2 latency and FP32 issue (242
// CTAs of 640 threads, 1.7 times the tile's cells); 1.8 us a step against 8.2 with a launch
// per Heun stage (Dirichlet) and 6.2 for the per-tile kernel (periodic).
template <int EX, int EY, int S, int R>
struct DnsSteps {
    static constexpr int HALO = 2 * S, TX = EX - 2 * HALO, TY = EY - 2 * HALO, NT = EX * (EY / R);
    static_assert(EX % 32 == 0 && EY % R == 0 && NT <= 1024 && TX > 0 && TY > 0, "whole strips");
};
template <int EX, int EY, int S, int R, bool DIR>
__global__ void __launch_bounds__(DnsSteps<EX, EY, S, R>::NT)
k_dns_steps(int nf, const float *uin, const float *__restrict__ psi, float *uout,
            float cA, float cD, int steps, float ul, float ur)
{
    using D = DnsSteps<EX, EY, S, R>;
    __shared__ float A[EY * EX], Bf[EY * EX];
    const int x = threadIdx.x % EX, y0 = threadIdx.x / EX * R;
    const int gx0 = (int)blockIdx.x * D::TX - D::HALO + x, gy0 = (int)blockIdx.y * D::TY - D::HALO + y0;
    auto wrap = [&](int i) { return ((i % nf) + nf) % nf; };
    const int gx = wrap(gx0);
    const bool held = DIR && (gx0 == 0 || gx0 == nf);
    float u[R], s[R], pa[R], pb[R];              // u, stage value, psiS - psiN, psiE - psiW
    {
        const int ge = gx + 1 == nf ? 0 : gx + 1, gw = gx == 0 ? nf - 1 : gx - 1;
        float pc[R + 2];
#pragma unroll
        for (int r = -1; r <= R; ++r) pc[r + 1] = psi[(long long)wrap(gy0 + r) * nf + gx];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const long long row = (long long)wrap(gy0 + r) * nf;
            pa[r] = pc[r] - pc[r + 2];
            pb[r] = psi[row + ge] - psi[row + gw];
        }
        chain_wait();
#pragma unroll
        for (int r = 0; r < R; ++r) {
            u[r] = !held ? uin[(long long)wrap(gy0 + r) * nf + gx] : (gx0 == 0 ? ul : ur);
            A[(y0 + r) * EX + x] = u[r];
        }
    }
    __syncthreads();
    const int xw = x > 0 ? x - 1 : 0, xe = x < EX - 1 ? x + 1 : EX - 1;
    const int ym = y0 > 0 ? y0 - 1 : 0, yp = y0 + R < EY ? y0 + R : EY - 1;
    // g = x + dt f(x) of this thread's cells c, the field in X
    auto stage = [&](const float *X, const float (&c)[R], float (&g)[R]) {
        const float below = X[ym * EX + x], above = X[yp * EX + x];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const float W = X[(y0 + r) * EX + xw], E = X[(y0 + r) * EX + xe];
            const float N = r + 1 < R ? c[(r + 1) % R] : above, B = r > 0 ? c[(r + R - 1) % R] : below;
            float t = pa[r] * (E - W);
            t = fmaf(pb[r], N - B, t);
            const float lap = fmaf(-4.0f, c[r], (E + W) + (N + B));
            g[r] = fmaf(cA, t, fmaf(cD, lap, c[r]));
        }
    };
    for (int k = 0; k < steps; ++k) {
        float g[R];
        // rows 2k+1 .. EY-2-2k are valid after this stage
        if (y0 + R > 2 * k + 1 && y0 < EY - 1 - 2 * k) {
            stage(A, u, g);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                s[r] = held ? u[r] : g[r];
                Bf[(y0 + r) * EX + x] = s[r];
            }
        }
        __syncthreads();
        if (y0 + R > 2 * k + 2 && y0 < EY - 2 - 2 * k) {
            stage(Bf, s, g);
#pragma unroll
            for (int r = 0; r < R; ++r) {
                u[r] = held ? u[r] : 0.5f * (u[r] + g[r]);
                A[(y0 + r) * EX + x] = u[r];
            }
        }
        __syncthreads();
    }
    if (x >= D::HALO && x < D::HALO + D::TX && gx0 < nf)
#pragma unroll
        for (int r = 0; r < R; ++r)
            if (y0 + r >= D::HALO && y0 + r < D::HALO + D::TY && gy0 + r < nf)
                uout[(long long)(gy0 + r) * nf + gx0] = u[r];
}

// FP64 Dirichlet runs.  What bounds them is FP64 issue (2 operations a clock and SM), so the
// step is written with as few as possible: with A = dt f's linear part, Heun's step of this
// linear problem is u + A u + A^2 u / 2 = u + A' (s), s = sqrt2 u + A' u, A' = A / sqrt2, and
//   A' x = aE xE + aW xW + aN xN + aS xS - 4 d x,   d = dt kappa / (sqrt2 h^2),
//   aE, aW = d +- c1, aN, aS = d +- c2,  c1, c2 = dt / (4 sqrt2 h^2) (psiS - psiN, psiE - psiW):
// 5 operations a cell and stage, none of them a conversion (aE and aN come from arrays formed
// once per run; 12 operations and 4 conversions a cell and stage before).  512^2: 8.9 us a step
// against 24.7 with a launch per stage.  The boundary values enter the first stage scaled by sqrt2.
// Grids above kDirCoefMax^2 (1 GB of coefficients), and calls whose coefficients find no memory,
// form them again in every step: 10 operations and 4 conversions more per cell.
__global__ void k_dns_dir_coef(int nf, const float *__restrict__ psi, double cA, double d,
                               double *__restrict__ aE, double *__restrict__ aN)
{
    const long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (c >= (long long)nf * nf) return;
    const int a = (int)(c % nf), b = (int)(c / nf);
    const int bp = b + 1 == nf ? 0 : b + 1, bm = b == 0 ? nf - 1 : b - 1;
    const int ap = a + 1 == nf ? 0 : a + 1, am = a == 0 ? nf - 1 : a - 1;
    const long long row = (long long)b * nf;
    aE[c] = fma(cA, (double)psi[(long long)bm * nf + a] - (double)psi[(long long)bp * nf + a], d);
    aN[c] = fma(cA, (double)psi[row + ap] - (double)psi[row + am], d);
}

// One step of a 28 x TY tile per CTA, halo 2: a warp owns R rows of the 32 extended columns
// (east and west neighbours by shuffles), rows outside a stage's valid ones are skipped.
constexpr int kD64R = 2, kD64TX = 28;
template <int TY>
__global__ void __launch_bounds__(32 * (TY + 4) / kD64R)
k_dns_dir_step64(int nf, const double *uin, double *uout, const double *__restrict__ aEg,
                 const double *__restrict__ aNg, const float *__restrict__ psi, double cA, double d,
                 double ul, double ur, double ul_s, double ur_s)
{
    constexpr int R = kD64R, EY = TY + 4;
    __shared__ double A[EY * 32], Bf[EY * 32];
    const int x = threadIdx.x & 31, y0 = (threadIdx.x >> 5) * R;
    const int gx0 = (int)blockIdx.x * kD64TX - 2 + x, gy0 = (int)blockIdx.y * TY - 2 + y0;
    auto wrap = [&](int i) { return ((i % nf) + nf) % nf; };
    const int gx = wrap(gx0);
    const bool held = gx0 == 0 || gx0 == nf;
    const double two_d = 2.0 * d, m4d = -4.0 * d;
    double u[R], aE[R], aN[R], aW[R], aS[R], s[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int gy = wrap(gy0 + r);
        const long long row = (long long)gy * nf, c = row + gx;
        if (aEg) {
            aE[r] = aEg[c];
            aN[r] = aNg[c];
        } else {                                        // as k_dns_dir_coef
            const int gp = gy + 1 == nf ? 0 : gy + 1, gm = gy == 0 ? nf - 1 : gy - 1;
            const int ap = gx + 1 == nf ? 0 : gx + 1, am = gx == 0 ? nf - 1 : gx - 1;
            aE[r] = fma(cA, (double)psi[(long long)gm * nf + gx] - (double)psi[(long long)gp * nf + gx], d);
            aN[r] = fma(cA, (double)psi[row + ap] - (double)psi[row + am], d);
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) { aW[r] = two_d - aE[r]; aS[r] = two_d - aN[r]; }
    chain_wait();
#pragma unroll
    for (int r = 0; r < R; ++r) {
        u[r] = !held ? uin[(long long)wrap(gy0 + r) * nf + gx] : (gx0 == 0 ? ul : ur);
        A[(y0 + r) * 32 + x] = u[r];
    }
    __syncthreads();
    // acc + A' x without the centre term, c this thread's rows of the field in X
    auto ring = [&](const double *X, const double (&c)[R], int r, double acc) {
        const double E = __shfl_down_sync(0xffffffffu, c[r], 1), W = __shfl_up_sync(0xffffffffu, c[r], 1);
        const double N = r + 1 < R ? c[(r + 1) % R] : X[(y0 + R < EY ? y0 + R : EY - 1) * 32 + x];
        const double B = r > 0 ? c[(r + R - 1) % R] : X[(y0 > 0 ? y0 - 1 : 0) * 32 + x];
        acc = fma(aE[r], E, acc);
        acc = fma(aW[r], W, acc);
        acc = fma(aN[r], N, acc);
        return fma(aS[r], B, acc);
    };
    // stage 1 on rows 1 .. EY-2 (the strips at the rim compute theirs with a clamped row)
    const double centre = 1.4142135623730951 + m4d;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const double g = ring(A, u, r, centre * u[r]);
        s[r] = !held ? g : (gx0 == 0 ? ul_s : ur_s);
        Bf[(y0 + r) * 32 + x] = s[r];
    }
    __syncthreads();
    // stage 2 and the store: the strips of the tile's own rows
    if (y0 < 2 || y0 >= EY - 2) return;
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const double g = ring(Bf, s, r, fma(m4d, s[r], u[r]));
        if (x >= 2 && x < 2 + kD64TX && gx0 < nf && gy0 + r < nf)
            uout[(long long)(gy0 + r) * nf + gx0] = held ? u[r] : g;
    }
}

// max over the grid of |v1| + |v2| (non-negative floats order like their bit patterns)
__global__ void k_dns_vmax(int nf, const float *psi, float ax, unsigned *out)
{
    float m = 0.f;
    const long long n2 = (long long)nf * nf;
    for (long long c = blockIdx.x * (long long)blockDim.x + threadIdx.x; c < n2;
         c += (long long)gridDim.x * blockDim.x) {
        const int b = (int)(c / nf), a = (int)(c % nf);
        const int bp = b + 1 == nf ? 0 : b + 1, bm = b == 0 ? nf - 1 : b - 1;
        const int ap = a + 1 == nf ? 0 : a + 1, am = a == 0 ? nf - 1 : a - 1;
        const float v1 = (psi[(long long)bm * nf + a] - psi[(long long)bp * nf + a]) * ax;
        const float v2 = (psi[(long long)b * nf + ap] - psi[(long long)b * nf + am]) * ax;
        m = fmaxf(m, fabsf(v1) + fabsf(v2));
    }
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out, __float_as_uint(m));
}

// Box average onto the macro grid; box[j*N+i] = FP64 sum of the box.  W warps a box, PER nodes a
// lane at a time, each read once.  An SM issues 2 FP64 operations a clock: converting and adding
// every node in FP64 took 8 times as long as reading it.  So up to T PER nodes at a time are
// added as integers: with E the largest exponent of the n <= 2^bits nodes and shift = 38 - bits,
// each becomes its 24-bit significand in units of 2^(E - 150 - shift), so that n of them fit
// 62 bits.  That is exact where every node but zeros is within 2^shift (2^26 at least) of the
// largest, and the sum is rounded once to FP64.  Nodes further apart, which integers would round to
// their unit, are added in FP64, as infinities and NaN are.  The 8 warps' FP64 work is left to one
// of them (a warp with one box takes as long as one with 8).  8192^2 onto 64^2, 128^2, 512^2: 288, 367, 2081 us
// for a CTA a box in FP64; 130, 136, 150 so (118, 122, 144 without looking for nodes too far
// apart, each of them then off by up to 2^-50 of the largest); 311, 314, 359 where every box has such
// nodes (reading them once: 40).  What bounds it: the integer operations, about 27 a node.
template <int W, int PER>
__global__ void __launch_bounds__(256) k_coarse(int nf, const float *__restrict__ u, int N, float *U,
                                                double *box, int bits)
{
    constexpr int T = 32 * W, BOXES = 8 / W;          // threads per box, boxes per CTA
    __shared__ unsigned tops[8], lows[8];
    __shared__ long long accs[8];
    __shared__ double sums[8];
    const int r = nf / N, n = r * r, t = threadIdx.x % T, warp = threadIdx.x >> 5, w0 = warp / W * W;
    const long long b = (long long)blockIdx.x * BOXES + threadIdx.x / T;
    const bool in = b < (long long)N * N;
    const int i = (int)(b % N), j = (int)(b / N), x0 = i * r - r / 2, y0 = j * r - r / 2;
    const int sx = T % r, sy = T / r, shift = 38 - bits;
    auto exponent = [](unsigned a) { return max(1, (int)(a >> 23)); };    // denormals: that of 2^-126
    // whether nodes of magnitudes low + 1 .. top (zeros aside) fit integers exactly
    auto integers = [&](unsigned top, unsigned low) {
        return exponent(top) < 255 && exponent(top) - exponent(low + 1) <= shift;
    };
    // thread k < BOXES: the sum of the CTA's k-th box.  One chunk of nodes unless W = 8
    double total = 0.0;
    int x = t % r, y = t / r;
    for (int base = 0; base < (W < 8 ? 1 : n); base += T * PER) {
        // the lane's nodes: every T-th of the box's, row by row
        unsigned v[PER], top = 0, low = ~0u;              // low: the least magnitude - 1, zeros last
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            int gx = x0 + x, gy = y0 + y;
            gx = gx < 0 ? gx + nf : gx;                // a box reaches past the grid's start only
            gy = gy < 0 ? gy + nf : gy;
            v[k] = in && base + t + k * T < n ? __float_as_uint(__ldg(u + (long long)gy * nf + gx)) : 0u;
            x += sx;
            y += sy;
            if (x >= r) { x -= r; ++y; }
        }
#pragma unroll
        for (int k = 0; k < PER; ++k) {
            top = max(top, v[k] & 0x7fffffffu);
            low = min(low, (v[k] & 0x7fffffffu) - 1u);
        }
        top = __reduce_max_sync(0xffffffffu, top);
        low = __reduce_min_sync(0xffffffffu, low);
        if ((threadIdx.x & 31) == 0) { tops[warp] = top; lows[warp] = low; }
        if constexpr (W > 1) {
            __syncthreads();
#pragma unroll
            for (int w = 0; w < W; ++w) { top = max(top, tops[w0 + w]); low = min(low, lows[w0 + w]); }
        }
        const int E = exponent(top);
        long long acc = 0;
        if (integers(top, low)) {
#pragma unroll
            for (int k = 0; k < PER; ++k) {
                const int e = (v[k] >> 23) & 255, sh = shift - (E - max(1, e));
                const unsigned long long m = (v[k] & 0x7fffffu) | (e ? 0x800000u : 0u);
                const long long q = (long long)(m << (sh & 63));          // sh < 0 for zeros only
                acc += (v[k] >> 31) ? -q : q;
            }
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if ((threadIdx.x & 31) == 0) accs[warp] = acc;
        } else {
            double s = 0.0;
#pragma unroll
            for (int k = 0; k < PER; ++k) s += (double)__uint_as_float(v[k]);
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if ((threadIdx.x & 31) == 0) sums[warp] = s;
        }
        __syncthreads();
        if (threadIdx.x < BOXES) {
            unsigned tb = 0, lb = ~0u;
            long long a = 0;
            for (int w = 0; w < W; ++w) {
                tb = max(tb, tops[threadIdx.x * W + w]);
                lb = min(lb, lows[threadIdx.x * W + w]);
            }
            if (integers(tb, lb)) {
                for (int w = 0; w < W; ++w) a += accs[threadIdx.x * W + w];
                total += ldexp((double)a, exponent(tb) - 150 - shift);
            } else {
                for (int w = 0; w < W; ++w) total += sums[threadIdx.x * W + w];
            }
        }
        if constexpr (W == 8) __syncthreads();
    }
    const long long bo = (long long)blockIdx.x * BOXES + threadIdx.x;
    if (threadIdx.x < BOXES && bo < (long long)N * N) {
        U[bo] = (float)(total / ((double)r * r));
        if (box) box[bo] = total;
    }
}

__global__ void k_sum(int n, const double *x, double scale, double *out)
{
    __shared__ double red[32];
    double s = 0.0;
    for (int k = threadIdx.x; k < n; k += blockDim.x) s += x[k];
    s = block_sum(s, red);
    if (threadIdx.x == 0) *out = s * scale;
}

}  // namespace

// Which kernel takes an N x N grid: one CTA for the whole run up to 32^2 in FP32 and 16^2 in
// FP64 (where one SM's 2 FP64 operations a clock decide), tiles above.  A step, resident
// against tiles: FP32 0.83 us at 32^2 (tiles 1.1 at every side up to 128); FP64 4.05 us at 16^2
// and 6.5 at 20^2 (tiles 4.8 - 5.2 at sides 24 to 128).
static bool macro_resident(int N, int precision) { return N <= (precision == MLSD_FP64 ? 16 : 32); }
// tiles: 16 x 16 cells and 4 steps a launch in FP32; 16 x 8 cells and 1 step in FP64, where
// the recomputed halo costs more than a launch
constexpr int kTileX = 16, kTileY32 = 16, kSteps32 = 4, kTileY64 = 8, kSteps64 = 1;
static long long macro_tiles(int N, int precision)
{
    const int ty = precision == MLSD_FP64 ? kTileY64 : kTileY32;
    return (long long)((N + kTileX - 1) / kTileX) * ((N + ty - 1) / ty);
}
static long long macro_mass_blocks(int N, int precision)
{
    return std::max(((long long)N * N + 255) / 256, macro_tiles(N, precision));
}

// five fields, and with the mass record the tiles' shares of every step
size_t macro_scratch_bytes(int N, int precision, int nsteps, bool mass)
{
    const size_t rs = precision == MLSD_FP64 ? 8 : 4;
    const size_t NN = (size_t)N * N;
    if (macro_resident(N, precision)) return 0;
    const size_t parts = mass ? ((size_t)nsteps + 1) * macro_mass_blocks(N, precision) : 0;
    return 5 * NN * rs + 256 + parts * sizeof(double);
}

template <typename real, bool DIR>
static cudaError_t macro_run_t(int N, real *U, const double *K, double dt, int nsteps,
                               double *mass, void *scratch, cudaStream_t s, double ul, double ur)
{
    constexpr bool F64 = sizeof(real) == 8;
    constexpr int prec = F64 ? MLSD_FP64 : MLSD_FP32;
    const int NN = N * N, th = 256, nb = (NN + th - 1) / th;
    const double H = 2.0 * kPi / N;
    const real f = (real)(0.5 * dt / (H * H)), l = (real)ul, r = (real)ur;
    if (macro_resident(N, prec)) {
        const int threads = (NN + 31) / 32 * 32;
        count_launches(1);
        k_macro_resident<real, F64 ? 256 : 1024, DIR><<<1, threads, 2 * (size_t)NN * sizeof(real), s>>>(
            N, U, K, f, nsteps, mass, l, r);
        return cudaGetLastError();
    }
    real *co = static_cast<real *>(scratch), *V = co + 4 * (size_t)NN;
    constexpr int S = F64 ? kSteps64 : kSteps32, TY = F64 ? kTileY64 : kTileY32;
    const int launches = nsteps / S + (nsteps % S ? 1 : 0);
    // the tile launches ping-pong between U and V and end in U
    const bool start_in_V = launches & 1;
    count_launches(1);
    k_macro_prep<real><<<nb, th, 0, s>>>(N, K, f, co, U, start_in_V ? V : nullptr, DIR ? 1 : 0, l);
    double *part = reinterpret_cast<double *>(
        (reinterpret_cast<uintptr_t>(V + NN) + 255) & ~(uintptr_t)255);
    using T = MacroTile<real, kTileX, TY, S, DIR>;
    const dim3 grid((N + kTileX - 1) / kTileX, (N + TY - 1) / TY);
    const long long tiles = (long long)grid.x * grid.y, stride = macro_mass_blocks(N, prec);
    count_launches(launches + (mass ? 3 : 0));
    if (mass) k_mass_part<real><<<nb, th, 0, s>>>(NN, U, part);
    real *a = start_in_V ? V : U, *b = start_in_V ? U : V;
    for (long long k = 0; k < nsteps; k += S) {
        const cudaError_t e = launch_chained(
            k_macro_tile<real, kTileX, TY, S, DIR>, grid, (T::NT + 31) / 32 * 32, 0, k > 0, s, N, a, b, co,
            (int)std::min<long long>(S, nsteps - k), mass ? part + stride + (size_t)k * tiles : nullptr, r);
        if (e != cudaSuccess) return e;
        std::swap(a, b);
    }
    if (mass) {
        k_mass_final<<<1, 128, 0, s>>>(1, nb, part, H * H, mass);
        if (nsteps > 0)
            k_mass_final<<<(unsigned)((nsteps + 127LL) / 128), 128, 0, s>>>(nsteps, (int)tiles, part + stride, H * H, mass + 1);
    }
    return cudaGetLastError();
}

cudaError_t macro_run(int N, void *U, int precision, const double *K, double dt, int nsteps,
                      double *mass_dev, void *scratch, cudaStream_t s)
{
    if (precision == MLSD_FP64)
        return macro_run_t<double, false>(N, static_cast<double *>(U), K, dt, nsteps, mass_dev,
                                          scratch, s, 0.0, 0.0);
    return macro_run_t<float, false>(N, static_cast<float *>(U), K, dt, nsteps, mass_dev, scratch,
                                     s, 0.0, 0.0);
}

cudaError_t macro_run_dirichlet(int N, void *U, int precision, const double *K, double dt,
                                int nsteps, double ul, double ur, double *mass_dev, void *scratch,
                                cudaStream_t s)
{
    if (precision == MLSD_FP64)
        return macro_run_t<double, true>(N, static_cast<double *>(U), K, dt, nsteps, mass_dev,
                                         scratch, s, ul, ur);
    return macro_run_t<float, true>(N, static_cast<float *>(U), K, dt, nsteps, mass_dev, scratch,
                                    s, ul, ur);
}

cudaError_t macro_dt_max(int N, const double *K, double *max_dev, cudaStream_t s)
{
    count_launches(1);
    k_kmax<<<1, 1024, 0, s>>>(N * N, K, max_dev);
    return cudaGetLastError();
}

template <int DTY>
static cudaError_t dns_launch(int nf, const float *a, const float *psi, float *b, float ax, float kd,
                              float dt, bool overlap, cudaStream_t s)
{
    using T = DnsTile<DTY>;
    static bool attr = false;
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(&k_dns_step<DTY>),
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::SMEM);
        if (e != cudaSuccess) return e;
        attr = true;
    }
    return launch_chained(k_dns_step<DTY>, dim3(nf / DTX, nf / DTY), T::DTH, T::SMEM, overlap, s, nf, a, psi,
                          b, ax, kd, dt);
}

// The two tile counters of the persistent kernels.  A run zeroes both before its first launch, then
// its launches alternate them, each zeroing the other for its successor: a run does not depend on
// what ran before it, so that a captured one can be replayed (the counters kept between runs by
// the host were frozen into a graph: a replay could start on a used counter and leave tiles out).
// The memset costs a run about 2 us, a step of these kernels takes 10 and more.
struct DnsQueue {
    int *counters = nullptr;
    int which = 0;
};
static cudaError_t dns_queue(DnsQueue &out, cudaStream_t s)
{
    static std::mutex mu;
    static std::vector<int *> q;                    // by device
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(mu);
        if ((int)q.size() <= dev) q.resize(dev + 1, nullptr);
        if (!q[dev]) e = cudaMalloc((void **)&q[dev], 2 * sizeof(int));
        if (e != cudaSuccess) { q[dev] = nullptr; return e; }
        out.counters = q[dev];
    }
    out.which = 0;
    return cudaMemsetAsync(out.counters, 0, 2 * sizeof(int), s);
}

template <int DTY, int NBUF, bool PAIR = false>
static cudaError_t dns_launch_tma(int nf, const CUtensorMap &ma, const CUtensorMap &mp,
                                  const float *a, const float *psi, float *b, float ax, float kd,
                                  float dt, DnsQueue &queue, bool overlap, cudaStream_t s)
{
    using T = DnsTma<DTY, NBUF>;
    constexpr int DTH = DnsTile<DTY>::DTH;
    const void *fn = reinterpret_cast<const void *>(&k_dns_tma<DTY, NBUF, PAIR>);
    static std::mutex mu;
    static std::vector<int> per_sm;                 // resident CTAs per SM, by device
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    int res = 0;
    {
        std::lock_guard<std::mutex> lock(mu);
        if ((int)per_sm.size() <= dev) per_sm.resize(dev + 1, 0);
        if (per_sm[dev] == 0) {
            e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::SMEM);
            if (e == cudaSuccess)
                e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[dev], fn, DTH, T::SMEM);
            if (e != cudaSuccess) return e;
            if (per_sm[dev] < 1) return cudaErrorInvalidConfiguration;
        }
        res = per_sm[dev];
    }
    const long long ntiles = (long long)(nf / DTX) * (nf / DTY);
    const int grid = (int)std::min<long long>(ntiles, (long long)res * sms);
    const int which = queue.which;
    queue.which ^= 1;
    return launch_chained(k_dns_tma<DTY, NBUF, PAIR>, dim3((unsigned)grid), DTH, T::SMEM, overlap, s, ma, mp, nf,
                          a, psi, b, ax, kd, dt, queue.counters, which);
}

// DNS kernel variants: per-tile CTAs staged by cp.async (tile height 64 rows, 2 CTAs/SM,
// or 32 rows, 4 CTAs/SM), or persistent CTAs fed by tensor copies (32 rows with one or
// two staging buffers, 64 rows with one; 32 rows with the f32x2 pair arithmetic).
// Picked once per process by timing each on the caller's grid;
// MLSD_DNS_TY = 64 | 32 | t32 | t32x2 | t64 | t32p pins one for the runs it is set for.
enum DnsKind { kCp64, kCp32, kTma32, kTma32x2, kTma64, kTma32p, kSteps, kDnsKinds };
static std::atomic<int> g_dns_choice{-1};        // the timed choice
static std::atomic<int> g_dns_last{-1};          // the kernel of the last run

static cudaError_t dns_launch_kind(int kind, int nf, const CUtensorMap *maps, int ia,
                                   const float *a, const float *psi, float *b, float ax, float kd,
                                   float dt, DnsQueue &queue, bool overlap, cudaStream_t s)
{
    switch (kind) {
    case kCp64: return dns_launch<64>(nf, a, psi, b, ax, kd, dt, overlap, s);
    case kCp32: return dns_launch<32>(nf, a, psi, b, ax, kd, dt, overlap, s);
    case kTma32: return dns_launch_tma<32, 1>(nf, maps[ia], maps[2], a, psi, b, ax, kd, dt, queue, overlap, s);
    case kTma32x2: return dns_launch_tma<32, 2>(nf, maps[ia], maps[2], a, psi, b, ax, kd, dt, queue, overlap, s);
    case kTma64: return dns_launch_tma<64, 1>(nf, maps[ia], maps[2], a, psi, b, ax, kd, dt, queue, overlap, s);
    case kTma32p:
        return dns_launch_tma<32, 1, true>(nf, maps[ia], maps[2], a, psi, b, ax, kd, dt, queue, overlap, s);
    }
    return cudaErrorInvalidValue;
}

// nsteps steps by k_dns_steps launches that ping-pong between u and u_tmp, ending in u
template <bool DIR>
static cudaError_t dns_multi(int nf, float *u, float *u_tmp, const float *psi, float cA, float cD,
                             int nsteps, float ul, float ur, cudaStream_t s)
{
    constexpr int EX = 64, EY = 40, S = 4, R = 4;
    using D = DnsSteps<EX, EY, S, R>;
    // an even number of launches, the steps spread evenly over them (one step: a copy back)
    int launches = nsteps / S + (nsteps % S ? 1 : 0);
    if ((launches & 1) && nsteps > 1) ++launches;
    const dim3 grid((unsigned)((nf + D::TX - 1) / D::TX), (unsigned)((nf + D::TY - 1) / D::TY));
    count_launches(launches);
    float *a = u, *b = u_tmp;
    for (int k = 0, done = 0; k < launches; ++k) {
        const int upto = (int)((long long)nsteps * (k + 1) / launches);
        const cudaError_t e = launch_chained(k_dns_steps<EX, EY, S, R, DIR>, grid, D::NT, 0, k > 0, s, nf, a, psi,
                                             b, cA, cD, upto - done, ul, ur);
        if (e != cudaSuccess) return e;
        done = upto;
        std::swap(a, b);
    }
    if (a != u)
        return cudaMemcpyAsync(u, a, (size_t)nf * nf * sizeof(float), cudaMemcpyDeviceToDevice, s);
    return cudaGetLastError();
}

// Grids up to this side take several steps a launch: 1024^2 in 5.6 us a step against 8.2 for
// k_dns_step<32>, the best of the others there; at 1536^2 that one takes 10.3 and the halo's
// recomputation would cost about 12.
constexpr int kDnsMultiMax = 1024;

cudaError_t dns_run(int nf, float *u, float *u_tmp, const float *psi, double kappa, double dt,
                    int nsteps, cudaStream_t s)
{
    const double h = 2.0 * kPi / nf;
    const float ax = (float)(1.0 / (2.0 * h));
    const float kd = (float)(kappa / (h * h));
    if (nf <= kDnsMultiMax && !std::getenv("MLSD_DNS_TY")) {
        g_dns_last = kSteps;
        return dns_multi<false>(nf, u, u_tmp, psi, (float)dt * ax * ax, (float)dt * kd, nsteps, 0.f, 0.f, s);
    }
    // tensor maps of u, u_tmp and psi; boxes of DLX x (DTY + 4), one map set per tile height
    CUtensorMap m32[3], m64[3];
    const bool tma = encode_f32_2d(&m32[0], u, nf, nf, DLX, 36) &&
                     encode_f32_2d(&m32[1], u_tmp, nf, nf, DLX, 36) &&
                     encode_f32_2d(&m32[2], psi, nf, nf, DLX, 36) &&
                     encode_f32_2d(&m64[0], u, nf, nf, DLX, 68) &&
                     encode_f32_2d(&m64[1], u_tmp, nf, nf, DLX, 68) &&
                     encode_f32_2d(&m64[2], psi, nf, nf, DLX, 68);
    auto maps_of = [&](int kind) -> const CUtensorMap * { return kind == kTma64 ? m64 : m32; };
    int kind = g_dns_choice;
    if (const char *env = std::getenv("MLSD_DNS_TY")) {
        const std::string v(env);
        kind = v == "32" ? kCp32 : v == "t32" ? kTma32 : v == "t32x2" ? kTma32x2
                   : v == "t64" ? kTma64 : v == "t32p" ? kTma32p : kCp64;
    }
    if (!tma && kind >= kTma32) kind = kCp32;
    if (kind < 0) {
        // nothing can be timed (nor the queue made) under capture: the per-tile kernel, for this run
        cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
        const cudaError_t e = cudaStreamIsCapturing(s, &cs);
        if (e != cudaSuccess) return e;
        if (cs != cudaStreamCaptureStatusNone) kind = kCp32;
    }
    DnsQueue queue;
    if (nsteps > 0 && tma && (kind < 0 || kind >= kTma32)) {
        const cudaError_t e = dns_queue(queue, s);
        if (e != cudaSuccess) return e;
    }
    if (kind < 0 && nsteps > 0) {
        // one trial step of each into u_tmp (u is not modified), best of two
        cudaEvent_t e0, e1;
        cudaEventCreate(&e0);
        cudaEventCreate(&e1);
        float best = 1e30f;
        for (int k = 0; k < (tma ? (int)kSteps : (int)kTma32); ++k) {
            float t = 1e30f;
            for (int rep = 0; rep < 3; ++rep) {
                cudaEventRecord(e0, s);
                cudaError_t e = dns_launch_kind(k, nf, maps_of(k), 0, u, psi, u_tmp, ax, kd,
                                                (float)dt, queue, false, s);
                cudaEventRecord(e1, s);
                if (e != cudaSuccess) return e;
                cudaEventSynchronize(e1);
                float ms = 0.f;
                cudaEventElapsedTime(&ms, e0, e1);
                if (rep > 0) t = std::min(t, ms);
            }
            count_launches(3);
            if (t < best) { best = t; kind = k; }
        }
        cudaEventDestroy(e0);
        cudaEventDestroy(e1);
        g_dns_choice = kind;
    }
    g_dns_last = kind;
    float *a = u, *b = u_tmp;
    int ia = 0;
    count_launches(nsteps);
    for (int st = 0; st < nsteps; ++st) {
        cudaError_t e = dns_launch_kind(kind, nf, maps_of(kind), ia, a, psi, b, ax, kd,
                                        (float)dt, queue, st > 0, s);
        if (e != cudaSuccess) return e;
        float *t = a; a = b; b = t;
        ia ^= 1;
    }
    if (a != u)
        return cudaMemcpyAsync(u, a, (size_t)nf * nf * sizeof(float), cudaMemcpyDeviceToDevice, s);
    return cudaGetLastError();
}

const char *dns_kernel_name()
{
    static const char *names[kDnsKinds] = {"k_dns_step<64>", "k_dns_step<32>", "k_dns_tma<32,1>",
                                           "k_dns_tma<32,2>", "k_dns_tma<64,1>",
                                           "k_dns_tma<32,1,pairs>", "k_dns_steps"};
    const int kind = g_dns_last;
    return kind < 0 ? "" : names[kind];
}

int dns_status_take(cudaStream_t s)
{
    int v = 0;
    const int zero = 0;
    if (cudaMemcpyFromSymbolAsync(&v, g_dns_status, sizeof(int), 0, cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaMemcpyToSymbolAsync(g_dns_status, &zero, sizeof(int), 0, cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return MLSD_ECUDA;
    return v;
}

cudaError_t launch_wait_check_tile(int *status, cudaStream_t s)
{
    count_launches(1);
    k_wait_check_tile<<<1, 32, 0, s>>>(status);
    return cudaGetLastError();
}

constexpr int kDirCoefMax = 8192;
size_t dns_dirichlet_scratch_bytes(int nf, int precision, int nsteps)
{
    return precision == MLSD_FP64 && nsteps > 0 && nf <= kDirCoefMax ? 2 * (size_t)nf * nf * sizeof(double) : 0;
}

cudaError_t dns_run_dirichlet(int nf, void *u, void *u_tmp, const float *psi, int precision,
                              double kappa, double dt, int nsteps, double ul, double ur, void *scratch,
                              cudaStream_t s)
{
    const double h = 2.0 * kPi / nf;
    const double cA = dt / (4.0 * h * h), cD = dt * kappa / (h * h);
    if (nsteps == 0) {
        count_launches(1);
        if (precision == MLSD_FP64)
            k_set_col0<double><<<(nf + 255) / 256, 256, 0, s>>>(nf, static_cast<double *>(u), ul);
        else
            k_set_col0<float><<<(nf + 255) / 256, 256, 0, s>>>(nf, static_cast<float *>(u), (float)ul);
        return cudaGetLastError();
    }
    if (precision != MLSD_FP64)
        return dns_multi<true>(nf, static_cast<float *>(u), static_cast<float *>(u_tmp), psi, (float)cA,
                               (float)cD, nsteps, (float)ul, (float)ur, s);
    double *aE = static_cast<double *>(scratch), *aN = aE ? aE + (size_t)nf * nf : nullptr;
    const double r2 = 0.70710678118654752440;
    const long long n2 = (long long)nf * nf;
    count_launches((aE ? 1 : 0) + (long long)nsteps);
    if (aE) k_dns_dir_coef<<<(unsigned)((n2 + 255) / 256), 256, 0, s>>>(nf, psi, r2 * cA, r2 * cD, aE, aN);
    // tiles of 32 rows where they give every SM one, else of 8 (an SM's FP64 rate decides)
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const unsigned gx = (unsigned)((nf + kD64TX - 1) / kD64TX);
    const bool tall = (long long)gx * ((nf + 31) / 32) >= sms;
    const int ty = tall ? 32 : 8, nt = 32 * (ty + 4) / kD64R;
    const dim3 grid(gx, (unsigned)((nf + ty - 1) / ty));
    const auto fn = tall ? k_dns_dir_step64<32> : k_dns_dir_step64<8>;
    const double sq2 = 1.4142135623730951;
    double *a = static_cast<double *>(u), *b = static_cast<double *>(u_tmp);
    for (int k = 0; k < nsteps; ++k) {
        e = launch_chained(fn, grid, nt, 0, k > 0, s, nf, a, b, aE, aN, psi, r2 * cA, r2 * cD, ul, ur, sq2 * ul,
                           sq2 * ur);
        if (e != cudaSuccess) return e;
        std::swap(a, b);
    }
    if (a != u) return cudaMemcpyAsync(u, a, (size_t)n2 * sizeof(double), cudaMemcpyDeviceToDevice, s);
    return cudaGetLastError();
}

cudaError_t dns_vmax(int nf, const float *psi, unsigned *vmax_bits, cudaStream_t s)
{
    const double h = 2.0 * kPi / nf;
    cudaError_t e = cudaMemsetAsync(vmax_bits, 0, sizeof(unsigned), s);
    if (e != cudaSuccess) return e;
    count_launches(1);
    k_dns_vmax<<<1024, 256, 0, s>>>(nf, psi, (float)(1.0 / (2.0 * h)), vmax_bits);
    return cudaGetLastError();
}

cudaError_t coarse_grain(int nf, const float *u, int N, float *U, double *mass_dev,
                         cudaStream_t s)
{
    double *box = mass_dev ? mass_dev + 1 : nullptr;
    count_launches(mass_dev ? 2 : 1);
    const int r = nf / N;
    int bits = 0;                                      // of a chunk's nodes: 4096 at most
    while (bits < 12 && (1 << bits) < r * r) ++bits;
    const long long boxes = (long long)N * N;
    if (r <= 16) k_coarse<1, 8><<<(unsigned)((boxes + 7) / 8), 256, 0, s>>>(nf, u, N, U, box, bits);
    else if (r <= 32) k_coarse<2, 16><<<(unsigned)((boxes + 3) / 4), 256, 0, s>>>(nf, u, N, U, box, bits);
    else k_coarse<8, 16><<<(unsigned)boxes, 256, 0, s>>>(nf, u, N, U, box, bits);
    if (mass_dev) {
        const double h = 2.0 * kPi / nf;
        k_sum<<<1, 1024, 0, s>>>(N * N, box, h * h, mass_dev);
    }
    return cudaGetLastError();
}

}  // namespace mlsd

// ---------------------------------------------------------------------------
// Coarse-graining without allocation.
//
// Callers that must not allocate device memory (code running inside a host
// callback or a memory-pool-free embedding, allocator-less runtimes, or code
// that has handed all device memory to its own pool) get a variant of
// mlsd_coarse_grain whose scratch -- the FP64 box sums and the mass -- lives
// in the file-scope array below.  It holds 1 + MLSD_NOALLOC_MAX_MACRO^2
// doubles (about 512 KiB) on every device that loads the library, until the
// process exits.  Host code may not use the array's name as a pointer (it is
// a host-side stand-in): its device address is looked up once per device with
// cudaGetSymbolAddress, with that device current, on the first call there.
namespace mlsd {
namespace {
constexpr int kNoallocMax = MLSD_NOALLOC_MAX_MACRO;
constexpr int kNoallocDevices = 64;
static __device__ __align__(256) double g_cg_scratch[1 + kNoallocMax * kNoallocMax];
std::mutex g_noalloc_mu;
double *g_noalloc_ptr[kNoallocDevices] = {};

cudaError_t noalloc_scratch(double **out)
{
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNoallocDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_cg_scratch);
        if (e != cudaSuccess) return e;
        g_noalloc_ptr[dev] = static_cast<double *>(p);
    }
    *out = g_noalloc_ptr[dev];
    return cudaSuccess;
}
}  // namespace
}  // namespace mlsd

extern "C" int mlsd_coarse_grain_noalloc(int nf, const float *u_dev, int n_macro, float *U_dev,
                                         double *mass_out_host, void *cuda_stream)
{
    using namespace mlsd;
    if (nf < 1 || n_macro < 1 || nf % n_macro || !u_dev || !U_dev) return MLSD_EINVAL;
    if (n_macro > kNoallocMax) return MLSD_EINVAL;          // scratch holds N <= 256 only
    cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
    double *scratch = nullptr;
    if (noalloc_scratch(&scratch) != cudaSuccess) return MLSD_ECUDA;
    // every box sum and the mass are overwritten by this call: nothing carries over
    cudaError_t e = coarse_grain(nf, u_dev, n_macro, U_dev, mass_out_host ? scratch : nullptr, s);
    if (e == cudaSuccess && mass_out_host)
        e = cudaMemcpyAsync(mass_out_host, scratch, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess && mass_out_host) e = cudaStreamSynchronize(s);
    return e == cudaSuccess ? MLSD_OK : MLSD_ECUDA;
}
