// The gridpoint side of the method (Introduction, item ii: the grid is used to solve for the
// Eulerian quantities): node fields for the particle step from gridpoint statistics.
//
//   * recovery: element gradients of the P1 mean fields, area-weighted to the nodes; the
//     Laplacian is the recovered divergence of the recovered gradient;
//   * k = <u_i u_i>/2, eps = k <omega> (the paragraph before Eq. 5), production
//     P = -<u_i u_j> d<U_i>/dx_j and S_omega = C_omega2 - C_omega1 P/eps (Eq. 6);
//   * G_ij from elliptic relaxation (the paragraph after Eq. 4): P1 finite elements for
//     wp_ij - L^2 lap wp_ij = -3/4 C0 eps delta_ij with wall values wp_ij = -4.5 eps n_i n_j,
//     L = CL max(k^1.5/eps, Ceta nu^0.75/eps^0.25) (L^2 averaged over each element's nodes),
//     solved by a conjugate gradient in FP64 (Jacobi, or a polynomial in it) on the four components at
//     once; G_ij = (wp_ij - eps delta_ij/2)/k and C0 eps = -2/3 (eps + <u_i u_j> G_ij) (the
//     k-consistency condition), or the simplified Langevin model;
//   * mean pressure (optional; Section "Governing equations", the projection on the grid): weak
//     form of lap p = -d_i d_j (<U_i><U_j> + <u_i u_j>) with its natural boundary condition and
//     zero mean, by the same CG; a fixed mean gradient is added.
// Every reduction (gradient averaging, matrix assembly, dot products) is a gather in a fixed
// order, so the results are bit-reproducible run to run.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <type_traits>
#include <vector>

#include "lpdf_internal.h"

namespace lpdf {

namespace {

// the kernels take the tables by value: a member with a copy constructor would run it at every launch (a
// vector of one entry per unknown took 11 us of host time at 100,489)
static_assert(std::is_trivially_copyable<Fem>::value, "Fem is a kernel argument");

constexpr int kDotThreads = 256;
constexpr int kCheckEvery = 8;   // CG iterations between convergence tests

template <class T>
cudaError_t upload(T** d, const std::vector<T>& h)
{
    cudaError_t e = cudaMalloc((void**)d, sizeof(T) * std::max<size_t>(1, h.size()));
    if (e != cudaSuccess || h.empty()) return e;
    return cudaMemcpy(*d, h.data(), sizeof(T) * h.size(), cudaMemcpyHostToDevice);
}

inline unsigned blocks(int64_t n, int t = 256) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------- recovery
// element gradient of m DOF fields (row stride ld): out[(e m + i) 2 + j] = d_j f_i
__global__ void elem_grad_kernel(const Fem F, const double* __restrict__ f, int m, int ld, double* __restrict__ out)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= F.E) return;
    const int d0 = F.edof[3 * e], d1 = F.edof[3 * e + 1], d2 = F.edof[3 * e + 2];
    const double* g = F.grad + 6 * e;
    for (int i = 0; i < m; ++i) {
        const double a = f[(size_t)d0 * ld + i], b = f[(size_t)d1 * ld + i], c = f[(size_t)d2 * ld + i];
        out[((size_t)e * m + i) * 2 + 0] = a * g[0] + b * g[2] + c * g[4];
        out[((size_t)e * m + i) * 2 + 1] = a * g[1] + b * g[3] + c * g[5];
    }
}

// area-weighted average of m element values to the DOFs: out[d ld + i], a thread per value. (1/area is
// kept with the mesh: an FP64 division per thread is 600 cycles of a pipe that takes one warp at a time.
// The surrogate's call on 100,489 nodes 236 -> 229 us without it.)
__global__ void recover_kernel(const Fem F, const double* __restrict__ ev, int m, double* __restrict__ out, int ld)
{
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t0 >= (int64_t)F.ndof * m) return;
    const int d = (int)(t0 / m), i = (int)(t0 - (int64_t)d * m);
    double s = 0.0;
    for (int t = F.de_ptr[d]; t < F.de_ptr[d + 1]; ++t) {
        const int e = F.de_el[t] / 3;
        s += F.area[e] * ev[(size_t)e * m + i];
    }
    out[(size_t)d * ld + i] = s * F.iarea[d];
}

// element divergences of the three recovered gradients g (6 per DOF: d/dx, d/dy of each): out[3 e + i]
__global__ void elem_div_kernel(const Fem F, const double* __restrict__ g, double* __restrict__ out)
{
    const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t0 >= 3 * (int64_t)F.E) return;
    const int e = (int)(t0 / 3), i = (int)(t0 - 3 * (int64_t)e);
    const double* gr = F.grad + 6 * (size_t)e;
    double s = 0.0;
    for (int a = 0; a < 3; ++a) {
        const size_t d = F.edof[3 * (size_t)e + a];
        s += g[6 * d + 2 * i] * gr[2 * a] + g[6 * d + 2 * i + 1] * gr[2 * a + 1];
    }
    out[t0] = s;
}

// ---------------------------------------------------------------- per-DOF statistics
// statistics rows (S0, means, central moments, <omega>, <phi>, ...) of the DOF's master node, and
// the squared relaxation length L^2, L = CL max(k^1.5/eps, Ceta nu^0.75/eps^0.25): once per DOF (an
// element averages its three), its powers as square roots. kol = Ceta nu^0.75
__global__ void dof_stats_kernel(const Fem F, const double* __restrict__ st, int nq, int ns, double CL, double kol,
                                 double* __restrict__ U, double* __restrict__ R, double* __restrict__ om,
                                 double* __restrict__ phi, double* __restrict__ k, double* __restrict__ eps,
                                 double* __restrict__ L2)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= F.ndof) return;
    const double* s = st + (size_t)F.dof_node[d] * nq;
    for (int i = 0; i < 3; ++i) U[3 * (size_t)d + i] = s[1 + i];
    for (int i = 0; i < 6; ++i) R[6 * (size_t)d + i] = s[4 + i];
    om[d] = s[10];
    for (int a = 0; a < ns; ++a) phi[(size_t)d * ns + a] = s[11 + a];
    const double kk = 0.5 * (s[4] + s[7] + s[9]);
    const double e = kk * s[10];
    k[d] = kk;
    eps[d] = e;
    if (L2) {
        const double ep = fmax(e, 1e-12), kp = fmax(kk, 0.0);
        const double L = CL * fmax(kp * sqrt(kp) / ep, kol / sqrt(sqrt(ep)));
        L2[d] = L * L;
    }
}

// ---------------------------------------------------------------- assembly
__global__ void elem_L2_kernel(const Fem F, const double* __restrict__ L2, double* __restrict__ L2e)
{
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= F.E) return;
    double s = 0.0;
    for (int a = 0; a < 3; ++a) s += L2[F.edof[3 * e + a]];
    L2e[e] = s / 3.0;
}

// A = M + sum_e L2_e K_e (fixed contribution order per CSR entry); diag = its diagonal
// (and the largest row sum of |D^-1 A| of the rows that are solved for, a bound of its spectrum)
__global__ void assemble_kernel(const Fem F, const double* __restrict__ L2e, double* __restrict__ A,
                                double* __restrict__ diag, double* __restrict__ lmax)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= F.ndof) return;
    double total = 0.0;
    for (int j = F.row[i]; j < F.row[i + 1]; ++j) {
        double s = 0.0;
        for (int t = F.cptr[j]; t < F.cptr[j + 1]; ++t) {
            const int c = F.cel[t];
            const int e = c / 9, a = (c / 3) % 3, b = c % 3;
            const double* g = F.grad + 6 * e;
            s += L2e[e] * (F.area[e] * (g[2 * a] * g[2 * b] + g[2 * a + 1] * g[2 * b + 1]));
        }
        A[j] = F.Mval[j] + s;
        total += fabs(A[j]);
        if (F.col[j] == i) diag[i] = A[j];
    }
    // positive values compare like their bits
    if (!F.wall[i]) atomicMax(reinterpret_cast<long long*>(lmax), __double_as_longlong(total / diag[i]));
}

// ---------------------------------------------------------------- batched PCG
// vectors are stored component-major: v[c n + i]

// y_c = A x_c of the relaxation's four components
__global__ void spmv_kernel(const Fem F, const double* __restrict__ A, const double* __restrict__ x, double* __restrict__ y)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= F.ndof) return;
    const size_t n = F.ndof;
    double s[4] = {0, 0, 0, 0};
    for (int t = F.row[i]; t < F.row[i + 1]; ++t) {
        const int j = F.col[t];
        const double a = A[t];
        for (int c = 0; c < 4; ++c) s[c] += a * x[c * n + j];
    }
    for (int c = 0; c < 4; ++c) y[c * n + i] = s[c];
}

// Jacobi-preconditioned CG on one or two systems of the mesh's pattern (the relaxation's four
// right-hand sides and the pressure's one) in ONE cooperative launch, all components side by side.
//
// What bounds it: the chain of dependent steps of an iteration, not bytes (the matrix is a few MB)
// and not the launch any more (five launches per iteration took 20-33 us). Measured on this GPU: a
// warp's FP64 instruction takes 65 cycles, dependent or not (an SM sub-partition works on one at a
// time, 0.5 lanes per cycle), a division 600, a load from L2 330, a store with a fence 780. So the
// kernels count FP64 instructions on the critical path, divide once per sum, and never fence:
// every value that another warp reads travels as one 16-byte word (value, epoch), stored and loaded
// whole; a reader polls until the epoch is the one it waits for. The sums' partials travel the same
// way and are added in a fixed order, so a run gives the same bits every time.
// A word is overwritten only after everyone has read it: the next z is stored when the sum p.Ap of
// this iteration is known, whose partials depend on every read of the present z, and likewise for
// the partials. Polls are bounded; a warp that gives up records it and ends, and so do then the
// others.
//
// Converged when ||r_c|| <= tol ||r_c(xref)|| for every c of a system (xref NULL: the start itself),
// tested every kCheckEvery iterations and at maxit; a converged system stops there, and so does one
// with a norm that is not finite, which is not converged.
constexpr int kCgComps = 5;                       // components at most
constexpr int kCgSmallRows = 2048, kCgDeg = 12;   // cg_small_kernel: rows, matrix entries per row at most
constexpr int kCgSmallUnits = kCgSmallRows / 32;
constexpr int kCgMaxThreads = 1024;               // cg_kernel
constexpr int kCheb = 16;                         // its polynomial's degree and range (below)
constexpr double kChebRatio = 256.0;
enum { kCgIts0 = 0, kCgIts1 = 1, kCgOk = 2, kCgError = 3, kCgOut = 4 };   // kCgOk: systems converged

struct CgArgs {
    int n, nc, nv0, wpc, maxit, slice;      // slice: matrix entries per CTA in shared memory (0: none fit)
    int mask0, mask1;
    const int *row, *col;
    const unsigned char* wall;
    const double *A0, *A1, *d0, *d1, *b0, *b1, *ref0, *ref1;
    double *x0, *x1;
    double* state;                          // 4 nc n (r, p, q, 1/diag of cg_kernel with several rows per thread)
    const int *lcol, *halo_ptr, *halo;      // cg_kernel: see Fem
    int width;                              // its rows and halo, at most
    const double* lmax0;                    // bounds of the spectra of D^-1 A (device) and D^-1 K
    double lmax1;
    double cheb[2 * kCheb + 1];             // for a spectrum up to 1: 1 / theta, then the two coefficients of every step
    double tol;
    unsigned long long epoch, epochp;       // of z and the partial sums, of zp
    ulonglong2 *z, *slots;                  // nc n words; the partial sums' words
    ulonglong2* zp;                         // 2 nc n words
    int polls, quit;                        // polls (of about 0.2 us) before a wait gives up; see Fem
    int* out;
};

__device__ __forceinline__ void word_store(ulonglong2* p, double v, unsigned long long epoch)
{
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "mov.b128 t, {%1, %2};\n\t"
        "st.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p), "l"(__double_as_longlong(v)), "l"(epoch)
        : "memory");
}
__device__ __forceinline__ ulonglong2 word_raw(const ulonglong2* p)
{
    ulonglong2 w;
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "ld.relaxed.gpu.global.b128 t, [%2];\n\t"
        "mov.b128 {%0, %1}, t;\n\t}"
        : "=l"(w.x), "=l"(w.y)
        : "l"(p)
        : "memory");
    return w;
}
// the word's value; ok stays set only if its epoch is the expected one
__device__ __forceinline__ double word_load(const ulonglong2* p, unsigned long long epoch, bool& ok)
{
    long long b;
    unsigned long long e;
    asm volatile(
        "{\n\t.reg .b128 t;\n\t"
        "ld.relaxed.gpu.global.b128 t, [%2];\n\t"
        "mov.b128 {%0, %1}, t;\n\t}"
        : "=l"(b), "=l"(e)
        : "l"(p)
        : "memory");
    ok = ok && e == epoch;
    return __longlong_as_double(b);
}

// neither infinite nor NaN, from the exponent (a comparison is an FP64 instruction: 65 cycles)
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

__device__ __forceinline__ double shfl_add(double v, int o) { return __dadd_rn(v, __shfl_down_sync(0xffffffffu, v, o)); }

// a / b correctly rounded, given y = 1 / b correctly rounded (Markstein 1990): three FP64
// instructions instead of a division
__device__ __forceinline__ double div_by(double a, double b, double y)
{
    const double q = __dmul_rn(a, y);
    return __fma_rn(__fma_rn(-q, b, a), y, q);
}

// ---- up to kCgSmallRows rows: a warp per 32 rows of a component, no CTA or grid barrier at all.
// Unit u of a component is the rows 256 (u / 8) + u % 8 + 8 lane, whose words lie side by side (a
// neighbouring row's is then mostly the same lane's of the next unit). Every warp polls the units'
// partial sums itself (at most two words per lane) and adds them as a 256-thread block tree and
// then block by block. It keeps the p of its rows' neighbours in registers and advances them
// (p = z + beta p) from the neighbours' z, so p never travels; the z words are polled together with
// the partials of r.z.
__device__ __forceinline__ double cg_small_sum(double v0, double v1, int nu, int nb)
{
    v0 = shfl_add(shfl_add(shfl_add(v0, 4), 2), 1);
    if (nu > 32) v1 = shfl_add(shfl_add(shfl_add(v1, 4), 2), 1);
    double sum = __shfl_sync(0xffffffffu, v0, 0);
    for (int b = 1; b < nb; ++b) {
        const double t = __shfl_sync(0xffffffffu, b < 4 ? v0 : v1, (8 * b) & 31);
        sum = __dadd_rn(sum, t);
    }
    return sum;
}

__device__ __forceinline__ double cg_small_total(const ulonglong2* s, int nu, int nb, unsigned long long epoch, int lane,
                                                 int polls, bool& alive)
{
    double v0, v1;
    bool ok;
    int tries = 0;
    do {
        ok = true;
        v0 = lane < nu ? word_load(s + lane, epoch, ok) : 0.0;
        v1 = lane + 32 < nu ? word_load(s + lane + 32, epoch, ok) : 0.0;
        ok = __all_sync(0xffffffffu, ok);
    } while (!ok && ++tries < polls);
    alive = alive && ok;
    return cg_small_sum(v0, v1, nu, nb);
}

__device__ __forceinline__ double warp_tree(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = shfl_add(v, o);
    return v;   // lane 0's
}

__global__ void __launch_bounds__(32) cg_small_kernel(const __grid_constant__ CgArgs a)
{
    const int lane = threadIdx.x, nb = (a.n + 255) / 256, nu = 8 * nb, polls = a.polls;
    const int c = blockIdx.x / nu, u = blockIdx.x - c * nu;
    const bool sys = c >= a.nv0;
    const int v = sys ? c - a.nv0 : c, c0 = sys ? a.nv0 : 0, c1 = sys ? a.nc : a.nv0;   // the system's components
    const size_t n = a.n;
    const int i = 256 * (u >> 3) + (u & 7) + 8 * lane;
    const bool live = i < a.n;
    const double* const A = sys ? a.A1 : a.A0;
    const double* const ref = sys ? a.ref1 : a.ref0;
    double* const x = (sys ? a.x1 : a.x0) + v * n;
    ulonglong2* const zw = a.z + (size_t)c * 256 * nb;
    // words of the partial sums: [p.Ap, r.z, r0.r0, r.r, r.r][component][unit]; r.r in two sets used in
    // turn, as the components of a system only meet at the tests
    auto slot = [&](int k, int cc) { return a.slots + ((size_t)k * kCgComps + cc) * kCgSmallUnits; };
    const bool fixed = live && (sys ? a.mask1 : a.mask0) && a.wall[i];
    const int rs = live ? a.row[i] : 0, deg = live ? a.row[i + 1] - rs : 0;
    const int wdeg = __reduce_max_sync(0xffffffffu, deg);
    int word[kCgDeg];                          // the words of the row's columns
    int self = -1;
    double av[kCgDeg], pn[kCgDeg], zn[kCgDeg];
    double y = 0.0, yref = 0.0;
#pragma unroll
    for (int t = 0; t < kCgDeg; ++t) {
        const int j = t < deg ? a.col[rs + t] : -1;
        word[t] = j >= 0 ? (j & ~255) + 32 * (j & 7) + ((j & 255) >> 3) : -1;
        self = j == i ? t : self;
        av[t] = t < deg && !fixed ? A[rs + t] : 0.0;
        pn[t] = 0.0;
        if (j >= 0) {
            y = __fma_rn(av[t], x[j], y);
            if (ref) yref = __fma_rn(av[t], ref[v * n + j], yref);
        }
    }
    const double b = live ? (sys ? a.b1 : a.b0)[v * n + i] : 0.0;
    const double diag = live ? (sys ? a.d1 : a.d0)[i] : 1.0, dinv = 1.0 / diag;
    double xv = live ? x[i] : 0.0;
    double r = fixed ? 0.0 : __dsub_rn(b, y);
    double z = div_by(r, diag, dinv), q = 0.0;
    unsigned long long epoch = a.epoch;
    bool alive = (int)blockIdx.x != a.quit;
    auto post = [&](int k, double value) {
        const double s = warp_tree(value);
        if (lane == 0) word_store(slot(k, c) + u, s, epoch);
    };
    ulonglong2* const mine = zw + 32 * u + lane;
    if (live) word_store(mine, z, epoch);
    const double rref = ref ? (fixed ? 0.0 : __dsub_rn(b, yref)) : r;
    post(1, __dmul_rn(r, z));
    post(2, __dmul_rn(rref, rref));
    post(3, __dmul_rn(r, r));
    // the sum of r.z, and the z of the row's columns into zn
    auto gather = [&]() {
        bool ok;
        int tries = 0;
        auto load = [&]() {
            ok = true;
#pragma unroll
            for (int t = 0; t < kCgDeg; ++t) zn[t] = word[t] >= 0 ? word_load(zw + word[t], epoch, ok) : 0.0;
        };
        load();
        const double sum = cg_small_total(slot(1, c), nu, nb, epoch, lane, polls, alive);
        while (!__all_sync(0xffffffffu, ok) && ++tries < polls) load();   // mostly there by now
        alive = alive && __all_sync(0xffffffffu, ok);
        return sum;
    };
    double rz = gather();
    double r0[4], beta = 0.0;
    bool broken = false, done = false;             // broken: a norm is not finite
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        r0[k] = c0 + k < c1 ? a.tol * sqrt(cg_small_total(slot(2, c0 + k), nu, nb, epoch, lane, polls, alive)) : 0.0;
        broken = broken || !finite_bits(r0[k]);
    }
    int it = 0, set = 3;
    for (; alive; ++it) {
        if (it % kCheckEvery == 0 || it >= a.maxit) {
            done = true;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (c0 + k < c1) {
                    const double rr = cg_small_total(slot(set, c0 + k), nu, nb, epoch, lane, polls, alive);
                    if (!(sqrt(rr) <= r0[k])) done = false;
                    broken = broken || !finite_bits(rr);
                }
            done = done && !broken;
            if (!alive || done || broken || it >= a.maxit) break;
            set = 7 - set;
        }
        // p of the row and its neighbours, q = A p
        q = 0.0;
        double p = 0.0;
        auto advance = [&](int t) {
            pn[t] = __fma_rn(beta, pn[t], zn[t]);
            q = __fma_rn(av[t], pn[t], q);
            p = self == t ? pn[t] : p;
        };
#pragma unroll
        for (int t = 0; t < 7; ++t) advance(t);   // an interior row of a triangulation: 7 on average
        if (wdeg > 7) {
            advance(7);
            advance(8);
            if (wdeg > 9)
#pragma unroll
                for (int t = 9; t < kCgDeg; ++t) advance(t);
        }
        ++epoch;
        post(0, __dmul_rn(p, q));
        const double pq = cg_small_total(slot(0, c), nu, nb, epoch, lane, polls, alive);
        const double alpha = pq != 0.0 ? rz / pq : 0.0;
        r = __fma_rn(-alpha, q, r);
        z = div_by(r, diag, dinv);
        if (live) word_store(mine, z, epoch);
        post(1, __dmul_rn(r, z));
        if ((it + 1) % kCheckEvery == 0 || it + 1 >= a.maxit) post(set, __dmul_rn(r, r));
        xv = __fma_rn(alpha, p, xv);
        asm volatile("" : "+d"(rz));   // the reciprocal for beta is formed here, while the sum travels
        const double yrz = 1.0 / rz;
        const double rznew = gather();
        beta = rz != 0.0 ? div_by(rznew, rz, yrz) : 0.0;
        rz = rznew;
    }
    if (!alive) {
        if (lane == 0) atomicExch(a.out + kCgError, 1);
        return;
    }
    if (live) x[i] = xv;
    if (v == 0 && u == 0 && lane == 0) {
        a.out[sys ? kCgIts1 : kCgIts0] = it;
        if (done) atomicAdd(a.out + kCgOk, 1);
    }
}

// The preconditioner of cg_kernel with one row per thread and the matrix in shared memory: kCheb steps of
// the Chebyshev iteration for D^-1 A z = D^-1 r on [lmax / kChebRatio, lmax] (Golub & Varga 1961), lmax a
// Gershgorin bound: a fixed symmetric positive polynomial in D^-1 A. A step has no sum over the grid: a
// CTA stores its rows' z as words, polls the words of its halo (the other CTAs' rows that its rows refer
// to) into shared memory, and gathers from there after a barrier of the component's warps. What bounds it
// is that trip through L2 and the FP64 pipe (a dozen instructions of 65 cycles a warp): 2.4 us a step
// with the pressure alone at work, 6.5 with all five components. (Every thread polling its row's columns
// itself, up to ten words, was twice as slow.) Two buffers are used in turn: a thread overwrites what it
// stored two steps ago, which its neighbours' CTAs read before they stored what its own has read since;
// the pattern is symmetric. 25,351 nodes: the relaxation 16 iterations instead of 176, the pressure 64
// instead of 740, the solve 3.94 ms instead of 7.44; error against a 64-bit direct solve 2.5e-8 as before.
// In FP32 the solve took 2.65 ms, but the matrix overflows from a relaxation length of 2e19 on, and the
// call computes in FP64. (degree, ratio) = (8, 64) 4.41 ms, (12, 144) 4.37, (14, 196) 3.88, (16, 256) 3.94,
// (20, 400) 4.28; 2,976 nodes 2.31, 2.27, 2.23, 2.47, 2.51 ms, without it 3.95; 112,000 nodes, the pressure
// alone 11.2, 10.9, 10.6, 10.4, 10.2 ms.

// ---- any number of rows. CTA b owns the rows [n b / G, n (b + 1) / G) of every component; a warp
// works on one component (wpc warps each), a lane on one row, so neighbouring lanes gather
// neighbouring rows. kOne: at most one row per thread, so x, r, p, q and 1/diag stay in registers
// for the whole solve; otherwise they live in global memory (touched by their thread alone). Only z
// is read by other CTAs: A p is carried along by q = A z + beta q, so p never travels.
// kSmem: the CTA's slice of the matrix is staged in shared memory once. With both (up to 29,184 rows of
// the five components, 145,920 of the pressure alone) z = P(D^-1 r) as above, otherwise z = r/diag.
// A sum goes over the CTA's lanes to one word per CTA; one warp of one CTA per value collects the
// words, divides, and publishes the coefficient, which every CTA polls: two trips through L2. (All
// CTAs polling all words is one trip, but 152 x 152 polls of the same few lines took 12 us per
// iteration.) kCgTasks warps of a CTA do nothing else; meanwhile the others gather the neighbours'
// new z and form A z, which does not need beta.
constexpr int kCgTasks = 2;
struct CgShared {
    double red[3][kCgMaxThreads / 32 - kCgTasks][32];   // the threads' values
    double res[3][8];            // published sums
    double coef[8];              // alpha or beta of every component
    double rz[8];                // the collector's copy
    double r0[8], rr[8];
    unsigned active;             // components still iterating
    int stop, fail;
    int lost;                    // a wait of the CTA gave up: its others poll once more only
    double il[2];                // per system: 1 / the bound of its spectrum
};

constexpr int kCgPoll = 5;   // words polled at once by a lane

// The grid sums of `nval` values of every active component, by the task warps (w of kCgTasks); mode
// 0: res only; 1: coef = alpha = rz / sum; 2: value 0 is r.z, coef = beta. Words: partials
// [3][kCgComps][G] and published [2][3][kCgComps], in two sets used in turn.
__device__ __forceinline__ void cg_exchange(const CgArgs& a, CgShared& s, int w, int nval, int set,
                                            unsigned long long epoch, int mode)
{
    const int lane = threadIdx.x & 31, polls = a.polls;
    const int G = gridDim.x;
    const bool lost = s.lost;
    ulonglong2* const part = a.slots + (size_t)set * 3 * kCgComps * G;
    ulonglong2* const pub = a.slots + 2 * (size_t)3 * kCgComps * G + set * 3 * kCgComps * 2;
    for (int t = w; t < nval * a.nc; t += kCgTasks) {
        const int k = t / a.nc, c = t - k * a.nc;
        if (!((s.active >> c) & 1u)) continue;
        double v = s.red[k][c * a.wpc][lane];
        for (int q = 1; q < a.wpc; ++q) v = __dadd_rn(v, s.red[k][c * a.wpc + q][lane]);
        v = warp_tree(v);
        if (lane == 0) word_store(part + (size_t)t * G + blockIdx.x, v, epoch);
    }
    for (int t = w; t < nval * a.nc; t += kCgTasks) {
        const int k = t / a.nc, c = t - k * a.nc;
        if (!((s.active >> c) & 1u) || blockIdx.x != t % G) continue;
        double sum = 0.0;
        bool got = true;
        const double y = mode == 2 && k == 0 ? 1.0 / s.rz[c] : 0.0;
        for (int j0 = lane; j0 < G; j0 += 32 * kCgPoll) {
            double v[kCgPoll];
            bool ok;
            int tries = got && !lost ? 0 : polls;
            do {
                ok = true;
#pragma unroll
                for (int q = 0; q < kCgPoll; ++q)
                    v[q] = j0 + 32 * q < G ? word_load(part + (size_t)t * G + j0 + 32 * q, epoch, ok) : 0.0;
            } while (!ok && ++tries < polls);
            got = got && ok;
#pragma unroll
            for (int q = 0; q < kCgPoll; ++q) sum = __dadd_rn(sum, v[q]);
        }
        got = __all_sync(0xffffffffu, got);
        if (!got) s.fail = 1;
        sum = warp_tree(sum);
        if (lane == 0 && got) {   // (a sum that lacks a part is not published)
            double coef = 0.0;
            if (mode == 1) coef = sum != 0.0 ? s.rz[c] / sum : 0.0;
            if (mode == 2 && k == 0) coef = s.rz[c] != 0.0 ? div_by(sum, s.rz[c], y) : 0.0;
            word_store(pub + 2 * t, coef, epoch);
            word_store(pub + 2 * t + 1, sum, epoch);
        }
    }
    // lanes 2 q and 2 q + 1 poll this warp's q-th task
    const int t = w + kCgTasks * (lane >> 1);
    const int k = t / a.nc, c = t - k * a.nc;
    if (t < nval * a.nc && ((s.active >> c) & 1u)) {
        bool ok;
        double v;
        int tries = lost ? polls : 0;
        do {
            ok = true;
            v = word_load(pub + 2 * t + (lane & 1), epoch, ok);
        } while (!ok && ++tries < polls);
        if (!ok) s.fail = 1;
        if (lane & 1) s.res[k][c] = v;
        else if (mode && k == 0) s.coef[c] = v;
    }
}

template <bool kOne, bool kSmem>
__global__ void __launch_bounds__(kCgMaxThreads, 1) cg_kernel(const __grid_constant__ CgArgs a)
{
    extern __shared__ __align__(16) unsigned char dyn[];
    __shared__ CgShared s;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int task = wid - a.nc * a.wpc;          // >= 0: a task warp
    const int c = task >= 0 ? 0 : wid / a.wpc, sub = wid - c * a.wpc;
    const bool sys = c >= a.nv0;
    const int v = sys ? c - a.nv0 : c;
    const size_t n = a.n;
    const int lo = (int)((int64_t)a.n * blockIdx.x / gridDim.x), hi = (int)((int64_t)a.n * (blockIdx.x + 1) / gridDim.x);
    const int base = a.row[lo];
    const double* const gA = sys ? a.A1 : a.A0;
    double* const sA0 = reinterpret_cast<double*>(dyn);
    double* const sA1 = sA0 + (a.nv0 > 0 ? a.slice : 0);
    constexpr bool kPoly = kOne && kSmem;
    double* const sz = sA1 + (a.nc > a.nv0 ? a.slice : 0);                  // kPoly: [nc][2][width] of z
    int* const scol = reinterpret_cast<int*>(sz + (kPoly ? 2 * a.nc * a.width : 0));   // kPoly: indices into a z vector
    int* const shalo = scol + a.slice;                                      // kPoly: the other CTAs' rows read here
    int halo = 0;
    if (kSmem) {
        const int m = a.row[hi] - base;
        for (int t = threadIdx.x; t < m; t += blockDim.x) {
            if (a.nv0 > 0) sA0[t] = a.A0[base + t];
            if (a.nc > a.nv0) sA1[t] = a.A1[base + t];
            scol[t] = kPoly ? a.lcol[base + t] : a.col[base + t];
        }
    }
    if (kPoly) {
        halo = a.halo_ptr[blockIdx.x + 1] - a.halo_ptr[blockIdx.x];
        for (int t = threadIdx.x; t < halo; t += blockDim.x) shalo[t] = a.halo[a.halo_ptr[blockIdx.x] + t];
    }
    if (kPoly && threadIdx.x < 2)
        s.il[threadIdx.x] = 1.0 / (1.01 * (threadIdx.x ? a.lmax1 : (a.nv0 > 0 ? *a.lmax0 : 1.0)));
    if (threadIdx.x == 0) {
        s.active = (1u << a.nc) - 1u;
        s.stop = 0;
        s.fail = 0;
        s.lost = 0;
    }
    __syncthreads();
    const double* const sA = sys ? sA1 : sA0;
    unsigned long long epoch = a.epoch;
    const int polls = a.polls;
    const bool quit = (int)blockIdx.x == a.quit;
    bool bad = quit;
    // (A f) of a row; f(j) loads entry j, up to kW at once, until every word has its epoch. A CTA waits for a
    // lost word once, however many rows refer to lost ones.
    constexpr int kW = 10;
    auto row_dot = [&](int rs, int re, auto f) {
        double sum = 0.0;
        for (int t = rs; t < re; t += kW) {
            double zv[kW];
            bool ok;
            int tries = *(volatile int*)&s.lost ? polls : 0;
            do {
                ok = true;
#pragma unroll
                for (int u = 0; u < kW; ++u)
                    zv[u] = t + u < re ? f(kSmem && !kPoly ? scol[t + u - base] : __ldg(a.col + t + u), ok) : 0.0;
            } while (!ok && ++tries < polls);
            if (!ok) {
                bad = true;
                *(volatile int*)&s.lost = 1;
            }
#pragma unroll
            for (int u = 0; u < kW; ++u)
                if (t + u < re) sum = __fma_rn(kSmem ? sA[t + u - base] : __ldg(gA + t + u), zv[u], sum);
        }
        return sum;
    };
    // kPoly: fills the other CTAs' entries of a vector of the component (a thread at most every T-th, two at
    // once, the last one in place of one that is not there), then waits for all of its threads
    const int T = 32 * a.wpc, tid = 32 * sub + lane, width = a.width;
    auto gather_halo = [&](const ulonglong2* words, unsigned long long ep, double* zl) {
        for (int h = tid; h < halo; h += 2 * T) {
            const int h1 = min(h + T, halo - 1), j0 = shalo[h], j1 = shalo[h1];
            ulonglong2 w0 = word_raw(words + j0), w1 = word_raw(words + j1);
            int tries = bad ? polls : 0;
            while (w0.y != ep || w1.y != ep) {
                if (++tries >= polls) {
                    bad = true;
                    break;
                }
                w0 = word_raw(words + j0);
                w1 = word_raw(words + j1);
            }
            zl[hi - lo + h] = __longlong_as_double((long long)w0.x);
            zl[hi - lo + h1] = __longlong_as_double((long long)w1.x);
        }
        __syncwarp();
        asm volatile("bar.sync %0, %1;" ::"r"(1 + c), "r"(T) : "memory");
    };
    // sum + A times such a vector, eight entries of the row at once
    auto row_dot_local = [&](double sum, const double* zl, int rs, int re) {
        constexpr int kB = 8;
        for (int t = rs - base; t < re - base; t += kB) {
            double zz[kB], aa[kB];
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                const int at = min(t + u, re - base - 1);
                zz[u] = zl[scol[at]];
                aa[u] = sA[at];
            }
#pragma unroll
            for (int u = 0; u < kB; ++u) sum = t + u < re - base ? fma(aa[u], zz[u], sum) : sum;
        }
        return sum;
    };
    const int mask = sys ? a.mask1 : a.mask0;
    const double* const b = (sys ? a.b1 : a.b0) + v * n;
    const double* const ref0 = sys ? a.ref1 : a.ref0;
    const double* const ref = ref0 ? ref0 + v * n : nullptr;
    const double* const diag = sys ? a.d1 : a.d0;
    double* const x = (sys ? a.x1 : a.x0) + v * n;
    ulonglong2* const z = a.z + c * n;
    double* const st = a.state + 4 * c * n;
    const int first = task >= 0 ? hi : lo + 32 * sub + lane, stride = 32 * a.wpc;   // a task warp has no rows
    unsigned long long epochp = a.epochp;
    ulonglong2* const zp = a.zp + 2 * c * n;
    const bool mine = first < hi;
    // kPoly: z = P(D^-1 r) of the thread's row (all threads of the component take part; a fixed row's z
    // stays 0); d is the step before it is divided by the diagonal
    auto polynomial = [&](double r, double dinv, int rs, int re) {
        const double di = dinv * s.il[sys];
        double d = a.cheb[0] * r, zk = di * d;
#pragma unroll 1
        for (int k = 0; k < kCheb; ++k) {
            const unsigned long long ep = epochp + k;
            ulonglong2* const w = zp + (k & 1) * n;
            double* const zl = sz + (2 * c + (k & 1)) * width;
            if (mine) {
                word_store(w + first, zk, ep);
                zl[first - lo] = zk;
            }
            gather_halo(w, ep, zl);
            d = fma(a.cheb[1 + 2 * k], d, -a.cheb[2 + 2 * k] * row_dot_local(-r, zl, rs, re));
            zk = fma(di, d, zk);
        }
        epochp += kCheb;
        return zk;
    };
    // kOne: the row's state in registers
    double xv = 0.0, rv = 0.0, pv = 0.0, qv = 0.0, zv = 0.0, dinv = 0.0, sv = 0.0;
    int rs = 0, re = 0;
    double s0 = 0.0, s1 = 0.0, s2 = 0.0;
    for (int i = first; i < hi; i += stride) {
        rs = a.row[i];
        re = a.row[i + 1];
        const bool fixed = mask && a.wall[i];
        if (ref) {
            const double r = fixed ? 0.0 : b[i] - row_dot(rs, re, [&](int j, bool&) { return ref[j]; });
            s2 += r * r;
        }
        xv = x[i];
        rv = fixed ? 0.0 : b[i] - row_dot(rs, re, [&](int j, bool&) { return x[j]; });
        dinv = 1.0 / diag[i];
        zv = rv * dinv;
        if (!kPoly && !quit) word_store(z + i, zv, epoch);
        s0 += rv * zv;
        s1 += rv * rv;
        if (fixed) re = rs;   // its row of A p is zero
        if (!kOne) {
            st[i] = rv;
            st[n + i] = 0.0;
            st[2 * n + i] = 0.0;
            st[3 * n + i] = dinv;
        }
    }
    if (!ref) s2 = s1;
    // the sums of the threads' s0 (and s1, s2) over the grid; meanwhile, when `ahead` is set, A z
    auto zword = [&](int j, bool& have) { return word_load(z + j, epoch, have); };
    auto exchange = [&](int nval, int set, int mode, bool ahead) {
        if (task < 0) {
            s.red[0][wid][lane] = s0;
            if (nval > 1) s.red[1][wid][lane] = s1;
            if (nval > 2) s.red[2][wid][lane] = s2;
        }
        __syncthreads();
        if (task >= 0) cg_exchange(a, s, task, nval, set, epoch, mode);
        else if (kPoly && ahead) {
            // (the polynomial is done with its first buffer)
            double* const zl = sz + 2 * c * width;
            if (mine) zl[first - lo] = zv;
            gather_halo(z, epoch, zl);
            sv = row_dot_local(0.0, zl, rs, re);
        } else if (kOne && ahead && first < hi) sv = row_dot(rs, re, zword);
        if (bad) s.fail = 1;
        __syncthreads();
        return !s.fail;
    };
    bool ok = exchange(3, 1, 0, !kPoly);
    if (kPoly && ok) {
        s0 = 0.0;
        if (task < 0) {
            zv = polynomial(rv, dinv, rs, re);
            if (mine) {
                word_store(z + first, zv, epoch);
                s0 = rv * zv;
            }
        }
        ok = exchange(1, 0, 0, true);   // r.z into res[0]; r.r and |r_0|^2 stay in res[1], res[2]
    }
    if (threadIdx.x < a.nc) {
        s.rz[threadIdx.x] = s.res[0][threadIdx.x];
        s.rr[threadIdx.x] = s.res[1][threadIdx.x];
        s.r0[threadIdx.x] = sqrt(s.res[2][threadIdx.x]);
        s.coef[threadIdx.x] = 0.0;
    }
    __syncthreads();
    int its0 = a.maxit, its1 = a.maxit, conv = 0;   // thread 0's
    for (int it = 0; ok; ++it) {
        if (it % kCheckEvery == 0 || it >= a.maxit) {
            if (wid == 0) {
                const bool on = lane < a.nc && ((s.active >> lane) & 1u);
                const double rr = on ? s.rr[lane] : 0.0, limit = on ? a.tol * s.r0[lane] : 0.0;
                const unsigned broken = __ballot_sync(0xffffffffu, !finite_bits(rr) || !finite_bits(limit));
                const unsigned f = __ballot_sync(0xffffffffu, !(sqrt(rr) <= limit)) | broken;
                if (lane == 0) {
                    const unsigned m0 = (1u << a.nv0) - 1u, m1 = ((1u << a.nc) - 1u) & ~m0;
                    unsigned act = s.active;
                    if ((act & m0) && (!(f & m0) || (broken & m0))) { act &= ~m0; its0 = it; conv += !(f & m0); }
                    if ((act & m1) && (!(f & m1) || (broken & m1))) { act &= ~m1; its1 = it; conv += !(f & m1); }
                    s.active = act;
                    s.stop = act == 0u || it >= a.maxit;
                }
            }
            __syncthreads();
            if (s.stop) break;
        }
        const bool on = task < 0 && ((s.active >> c) & 1u);
        // r.r is only needed at the next test
        const bool test = (it + 1) % kCheckEvery == 0 || it + 1 >= a.maxit;
        s0 = 0.0;
        if (on) {
            const double beta = s.coef[c];
            if (kOne) {
                pv = __fma_rn(beta, pv, zv);
                qv = __fma_rn(beta, qv, sv);
                s0 = pv * qv;
            } else {
                for (int i = first; i < hi; i += stride) {
                    const int r0 = a.row[i], r1 = mask && a.wall[i] ? r0 : a.row[i + 1];
                    const double p = __fma_rn(beta, st[n + i], st[i] * st[3 * n + i]);
                    const double q = __fma_rn(beta, st[2 * n + i], row_dot(r0, r1, zword));
                    st[n + i] = p;
                    st[2 * n + i] = q;
                    s0 = __fma_rn(p, q, s0);
                }
            }
        }
        ++epoch;
        ok = exchange(1, 0, 1, false);
        if (!ok) break;
        s0 = s1 = 0.0;
        if (on) {
            const double alpha = s.coef[c];
            if (kOne) {
                rv = __fma_rn(-alpha, qv, rv);
                zv = kPoly ? polynomial(rv, dinv, rs, re) : rv * dinv;
                if (first < hi) {
                    word_store(z + first, zv, epoch);
                    s0 = rv * zv;
                    if (test) s1 = rv * rv;
                    xv = __fma_rn(alpha, pv, xv);
                }
            } else {
                for (int i = first; i < hi; i += stride) {
                    const double r = __fma_rn(-alpha, st[2 * n + i], st[i]), zz = r * st[3 * n + i];
                    st[i] = r;
                    word_store(z + i, zz, epoch);
                    s0 = __fma_rn(r, zz, s0);
                    s1 = __fma_rn(r, r, s1);
                    x[i] = __fma_rn(alpha, st[n + i], x[i]);
                }
            }
        }
        ok = exchange(test ? 2 : 1, 1, 2, on);
        if (threadIdx.x < a.nc) {
            s.rz[threadIdx.x] = s.res[0][threadIdx.x];
            if (test) s.rr[threadIdx.x] = s.res[1][threadIdx.x];
        }
    }
    if (!ok) {
        if (threadIdx.x == 0) atomicExch(a.out + kCgError, 1);
        return;
    }
    if (kOne && first < hi) x[first] = xv;
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.out[kCgIts0] = a.nv0 > 0 ? its0 : 0;
        a.out[kCgIts1] = a.nc > a.nv0 ? its1 : 0;
        a.out[kCgOk] = conv;
    }
}

// block partials of the sum of x, fixed order: a tree over 256 values
__global__ void sum_kernel(const double* __restrict__ x, int n, double* __restrict__ part)
{
    __shared__ double sh[kDotThreads];
    double s = 0.0;
    for (int i = blockIdx.x * kDotThreads + threadIdx.x; i < n; i += gridDim.x * kDotThreads) s += x[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int o = kDotThreads / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

constexpr size_t kCgSmemMax = 96 * 1024, kCgPolySmemMax = 192 * 1024;

// words of the partial sums (cg_small_kernel's, cg_kernel's with its published sums)
size_t cg_slot_words(int ctas)
{
    return std::max((size_t)5 * kCgComps * kCgSmallUnits, 2 * (size_t)3 * kCgComps * ctas + 2 * 3 * kCgComps * 2);
}

cudaError_t cg_configure()
{
    cudaError_t e = cudaFuncSetAttribute(cg_kernel<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCgPolySmemMax);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(cg_kernel<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kCgSmemMax);
    return e;
}

// ---------------------------------------------------------------- right-hand sides
// elliptic relaxation: sources wp^h (11, 12, 22, 33); wall values in x (the CG's start, whose
// interior is `prev`, or 0) and in xref (interior 0: the reference of the convergence test)
__global__ void er_setup_kernel(const Fem F, const double* __restrict__ eps, double C0, double* __restrict__ src,
                                double* __restrict__ x, const double* __restrict__ prev, double* __restrict__ xref)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= F.ndof) return;
    const size_t n = F.ndof;
    const double e = eps[d];
    const double n1 = F.normal[2 * d], n2 = F.normal[2 * d + 1];
    const double s = -0.75 * C0 * e;
    const bool w = F.wall[d];
    src[0 * n + d] = s;
    src[1 * n + d] = 0.0;
    src[2 * n + d] = s;
    src[3 * n + d] = s;
    const double wv[4] = {-4.5 * e * n1 * n1, -4.5 * e * n1 * n2, -4.5 * e * n2 * n2, 0.0};
    for (int c = 0; c < 4; ++c) {
        xref[c * n + d] = w ? wv[c] : 0.0;
        x[c * n + d] = w ? wv[c] : (prev ? prev[c * n + d] : 0.0);
    }
}

// T = <U><U> + <uu> in the plane: (T00, T01, T10, T11) per DOF
__global__ void pressure_T_kernel(const Fem F, const double* __restrict__ U, const double* __restrict__ R,
                                  double* __restrict__ T)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= F.ndof) return;
    const double u = U[3 * d], v = U[3 * d + 1];
    T[4 * d + 0] = u * u + R[6 * d + 0];
    T[4 * d + 1] = u * v + R[6 * d + 1];
    T[4 * d + 2] = u * v + R[6 * d + 1];
    T[4 * d + 3] = v * v + R[6 * d + 3];
}

// b_d = -sum_(e, a: edof(e, a) = d) area_e grad(l_a) . (div T)_e, gT = element gradients of T
__global__ void pressure_rhs_kernel(const Fem F, const double* __restrict__ gT, double* __restrict__ b)
{
    const int d = blockIdx.x * blockDim.x + threadIdx.x;
    if (d >= F.ndof) return;
    double s = 0.0;
    for (int t = F.de_ptr[d]; t < F.de_ptr[d + 1]; ++t) {
        const int e = F.de_el[t] / 3, a = F.de_el[t] % 3;
        const double* g = gT + (size_t)e * 8;
        const double div0 = g[0] + g[3];    // d_x T00 + d_y T01
        const double div1 = g[4] + g[7];    // d_x T10 + d_y T11
        const double* gr = F.grad + 6 * e;
        s += -F.area[e] * (gr[2 * a] * div0 + gr[2 * a + 1] * div1);
    }
    b[d] = s;
}

__global__ void subtract_mean_kernel(int n, const double* __restrict__ part, int nb, double* __restrict__ x)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double sum = 0.0;
    for (int b = 0; b < nb; ++b) sum += part[b];
    if (i < n) x[i] -= sum / n;
}

// every system converged and every wait got its word: CTA 0 counts the systems, but another CTA may have
// given up after its last sum went out, and left its rows of x unwritten
__device__ __forceinline__ bool cg_clean(const int* out, int systems)
{
    return out[kCgOk] == systems && out[kCgError] == 0;
}

// the converged solutions, kept as the next solve's start
__global__ void keep_solution_kernel(const int* __restrict__ cg_out, int systems, int n4, const double* __restrict__ wp,
                                     double* __restrict__ wp_prev, int n, const double* __restrict__ p,
                                     double* __restrict__ p_prev)
{
    if (!cg_clean(cg_out, systems)) return;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n4) wp_prev[i] = wp[i];
    if (i < n) p_prev[i] = p[i];
}

// ---------------------------------------------------------------- the output fields
__global__ void fields_kernel(const Fem F, int ns, int nfp, const double* __restrict__ U, const double* __restrict__ R,
                              const double* __restrict__ om, const double* __restrict__ phi,
                              const double* __restrict__ k, const double* __restrict__ eps,
                              const double* __restrict__ gU, const double* __restrict__ lapU,
                              const double* __restrict__ gp, const double* __restrict__ wp, int gmodel, double C0,
                              double Comega1, double Comega2, double dpdx0, double dpdy0,
                              const float* __restrict__ surr, const float* __restrict__ snorm,
                              const int* __restrict__ cg_out, int systems, float* __restrict__ out)
{
    const int nd = blockIdx.x * blockDim.x + threadIdx.x;
    if (nd >= F.N) return;
    if (cg_out && !cg_clean(cg_out, systems)) return;   // no solution: the caller's fields stay
    const int d = F.dof[nd];
    const size_t n = F.ndof;
    const double* r = R + 6 * (size_t)d;       // uu, uv, uw, vv, vw, ww
    const double* g = gU + 6 * (size_t)d;      // dU/dx, dU/dy, dV/dx, dV/dy, dW/dx, dW/dy
    const double kk = k[d], e = eps[d], Om = om[d];
    const double prod = -(r[0] * g[0] + r[1] * g[1] + r[1] * g[2] + r[3] * g[3] + r[2] * g[4] + r[4] * g[5]);
    const double Som = e > 1e-12 ? Comega2 - Comega1 * prod / e : Comega2;
    double G11, G12, G21, G22, G33, c0e;
    if (surr) {
        // the surrogate's targets: G_ij / <omega> and C_0 epsilon / (k <omega>), standardised
        double y[6];
        for (int j = 0; j < 6; ++j)
            y[j] = (double)surr[(size_t)nd * mlp::kOutP + j] * snorm[mlp::nTS + j] + snorm[mlp::nTM + j];
        G11 = Om * y[0];
        G12 = Om * y[1];
        G21 = Om * y[2];
        G22 = Om * y[3];
        G33 = Om * y[4];
        c0e = fmax(0.0, kk * Om * y[5]);
    } else if (gmodel == 1) {
        G11 = G22 = G33 = -(0.5 + 0.75 * C0) * Om;
        G12 = G21 = 0.0;
        c0e = C0 * e;
    } else {
        const double kc = fmax(kk, 1e-12);
        G11 = (wp[0 * n + d] - 0.5 * e) / kc;
        G12 = wp[1 * n + d] / kc;
        G22 = (wp[2 * n + d] - 0.5 * e) / kc;
        G33 = (wp[3 * n + d] - 0.5 * e) / kc;
        c0e = fmax(0.0, -2.0 / 3.0 * (e + r[0] * G11 + 2.0 * r[1] * G12 + r[3] * G22 + r[5] * G33));
        G21 = G12;
    }
    float* o = out + (size_t)nd * nfp;
    o[LPDF_F_U + 0] = (float)U[3 * d];
    o[LPDF_F_U + 1] = (float)U[3 * d + 1];
    o[LPDF_F_U + 2] = (float)U[3 * d + 2];
    for (int i = 0; i < 6; ++i) o[LPDF_F_DUDX + i] = (float)g[i];
    for (int i = 0; i < 3; ++i) o[LPDF_F_LAPU + i] = (float)lapU[3 * (size_t)d + i];
    o[LPDF_F_DPDX] = (float)(gp[2 * d] + dpdx0);
    o[LPDF_F_DPDX + 1] = (float)(gp[2 * d + 1] + dpdy0);
    o[LPDF_F_G11] = (float)G11;
    o[LPDF_F_G11 + 1] = (float)G12;
    o[LPDF_F_G11 + 2] = (float)G21;
    o[LPDF_F_G11 + 3] = (float)G22;
    o[LPDF_F_G11 + 4] = (float)G33;
    o[LPDF_F_C0EPS] = (float)c0e;
    o[LPDF_F_OMEGA] = (float)Om;
    o[LPDF_F_SOMEGA] = (float)Som;
    for (int a = 0; a < ns; ++a) o[LPDF_F_PHI0 + a] = (float)phi[(size_t)d * ns + a];
    for (int i = LPDF_F_PHI0 + ns; i < nfp; ++i) o[i] = 0.0f;
}

// ---------------------------------------------------------------- learned-surrogate inputs
// nearest wall point of every geometric node: distance, wall edge and position on it (the edges
// in order, each with its images one period to the left, in place and to the right; the first
// strictly nearest point wins)
__global__ void wall_distance_kernel(int N, const double* __restrict__ xy, const double* __restrict__ seg,
                                     const int* __restrict__ seg_off, const int* __restrict__ ncomp, double period,
                                     double* __restrict__ dist, int* __restrict__ wseg, double* __restrict__ wt)
{
    const int nd = blockIdx.x * blockDim.x + threadIdx.x;
    if (nd >= N) return;
    const double px = xy[2 * nd], py = xy[2 * nd + 1];
    double best = 1e300, bt = 0.0;
    const int c = ncomp[nd], s0 = seg_off[c], s1 = seg_off[c + 1];
    int bs = s0;
    const int ni = period > 0.0 ? 1 : 0;
    for (int s = s0; s < s1; ++s) {
        const double ax = seg[4 * s], ay = seg[4 * s + 1], tx = seg[4 * s + 2] - ax, ty = seg[4 * s + 3] - ay;
        const double tt = tx * tx + ty * ty;
        for (int im = -ni; im <= ni; ++im) {
            const double qx = px - ax - im * period, qy = py - ay;
            const double t = fmin(1.0, fmax(0.0, (qx * tx + qy * ty) / tt));
            const double dx = qx - t * tx, dy = qy - t * ty;
            const double d2 = dx * dx + dy * dy;
            if (d2 < best) {
                best = d2;
                bs = s;
                bt = t;
            }
        }
    }
    dist[nd] = s1 > s0 ? sqrt(best) : 0.0;
    wseg[nd] = bs;
    wt[nd] = bt;
}

// inputs: wall distance, log k, log <omega>, b11, b22, b12, II_b = b_ij b_ij with the anisotropy
// b_ij = <u_i u_j> / (2 k) - delta_ij / 3, and log(eps_w / eps) with eps_w the dissipation
// k <omega> interpolated linearly along the wall edge to the nearest wall point; targets (from node fields): G11, G12, G21,
// G22, G33 over <omega>, C_0 epsilon / (k <omega>) and the relaxed trace wp_ii over its local value
// -9/4 C_0 epsilon (wp_ii = k G_ii + 3 epsilon / 2)
__global__ void features_kernel(const Fem F, const double* __restrict__ stats, int nq,
                                const float* __restrict__ fields, int nfp, double C0, float* __restrict__ feat,
                                float* __restrict__ tgt)
{
    const int nd = blockIdx.x * blockDim.x + threadIdx.x;
    if (nd >= F.N) return;
    const double* st = stats + (size_t)F.dof_node[F.dof[nd]] * nq;
    const double uu = st[4], uv = st[5], uw = st[6], vv = st[7], vw = st[8], ww = st[9], Om = st[10];
    const double k = 0.5 * (uu + vv + ww);
    double eps_w = 0.0;
    const int comp = F.ncomp[nd];
    const bool walls = F.seg_off[comp + 1] > F.seg_off[comp];
    if (walls) {
        const int s = F.wseg[nd];
        const double t = F.wt[nd];
        const double* sa = stats + (size_t)F.dof_node[F.dof[F.segn[2 * s]]] * nq;
        const double* sb = stats + (size_t)F.dof_node[F.dof[F.segn[2 * s + 1]]] * nq;
        const double ea = 0.5 * (sa[4] + sa[7] + sa[9]) * sa[10], eb = 0.5 * (sb[4] + sb[7] + sb[9]) * sb[10];
        eps_w = (1.0 - t) * ea + t * eb;
    }
    double b11 = 0.0, b22 = 0.0, b33 = 0.0, b12 = 0.0, b13 = 0.0, b23 = 0.0;
    if (k > 1e-12) {
        const double ik = 0.5 / k;
        b11 = uu * ik - 1.0 / 3.0;
        b22 = vv * ik - 1.0 / 3.0;
        b33 = ww * ik - 1.0 / 3.0;
        b12 = uv * ik;
        b13 = uw * ik;
        b23 = vw * ik;
    }
    float* f = feat + (size_t)nd * mlp::kIn;
    f[0] = (float)F.wdist[nd];
    f[1] = (float)log(fmax(k, 1e-12));
    f[2] = (float)log(fmax(Om, 1e-12));
    f[3] = (float)b11;
    f[4] = (float)b22;
    f[5] = (float)b12;
    f[6] = (float)(b11 * b11 + b22 * b22 + b33 * b33 + 2.0 * (b12 * b12 + b13 * b13 + b23 * b23));
    f[7] = (float)(walls ? log(fmax(eps_w, 1e-12) / fmax(k * Om, 1e-12)) : 0.0);
    if (!tgt) return;
    const float* o = fields + (size_t)nd * nfp;
    const double Omc = fmax(Om, 1e-12), kc = fmax(k, 1e-12), e = k * Om;
    float* y = tgt + (size_t)nd * mlp::kOut;
    for (int j = 0; j < 5; ++j) y[j] = (float)((double)o[LPDF_F_G11 + j] / Omc);
    y[5] = (float)((double)o[LPDF_F_C0EPS] / (kc * Omc));
    const double tr = k * ((double)o[LPDF_F_G11] + (double)o[LPDF_F_G11 + 3] + (double)o[LPDF_F_G11 + 4]) + 1.5 * e;
    y[6] = (float)(e > 1e-12 ? tr / (-2.25 * C0 * e) : 1.0);
}

// {sum (a - b)^2, sum b^2} over the G_ij and C_0 epsilon columns (one block)
__global__ void fields_compare_kernel(const float* __restrict__ a, const float* __restrict__ b, int N, int nfp,
                                      double* __restrict__ out)
{
    __shared__ double sh[2][1024];
    double d2 = 0.0, b2 = 0.0;
    for (int i = threadIdx.x; i < N * 6; i += blockDim.x) {
        const size_t at = (size_t)(i / 6) * nfp + LPDF_F_G11 + i % 6;
        const double x = a[at], y = b[at];
        d2 += (x - y) * (x - y);
        b2 += y * y;
    }
    sh[0][threadIdx.x] = d2;
    sh[1][threadIdx.x] = b2;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + o];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + o];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        out[0] = sh[0][0];
        out[1] = sh[1][0];
    }
}

}  // namespace

// ------------------------------------------------------------------------- host side

cudaError_t fem_build(const double* node_xy, int N, const int32_t* tri, int E, const int32_t* tag,
                      const std::vector<int32_t>& master, const std::vector<int32_t>& node_comp, double period,
                      Fem** out)
{
    *out = nullptr;
    std::vector<int> dof(N), dof_node;
    std::vector<int> dof_of(N, -1);
    int ndof = 0;
    for (int i = 0; i < N; ++i)
        if (master[i] == i) {
            dof_of[i] = ndof++;
            dof_node.push_back(i);
        }
    for (int i = 0; i < N; ++i) dof[i] = dof_of[master[i]];
    std::vector<int> edof(3 * (size_t)E);
    std::vector<double> area(E), grad(6 * (size_t)E);
    for (int e = 0; e < E; ++e) {
        double x[3], y[3];
        for (int a = 0; a < 3; ++a) {
            edof[3 * e + a] = dof[tri[3 * e + a]];
            x[a] = node_xy[2 * tri[3 * e + a]];
            y[a] = node_xy[2 * tri[3 * e + a] + 1];
        }
        const double det = (x[1] - x[0]) * (y[2] - y[0]) - (y[1] - y[0]) * (x[2] - x[0]);
        area[e] = 0.5 * det;
        for (int a = 0; a < 3; ++a) {
            const int b = (a + 1) % 3, c = (a + 2) % 3;
            grad[6 * e + 2 * a] = (y[b] - y[c]) / det;
            grad[6 * e + 2 * a + 1] = (x[c] - x[b]) / det;
        }
    }
    // DOF -> incident (element, corner) pairs, in element order
    std::vector<int> de_ptr(ndof + 1, 0), de_el(3 * (size_t)E);
    for (int e = 0; e < E; ++e)
        for (int a = 0; a < 3; ++a) ++de_ptr[edof[3 * e + a] + 1];
    for (int d = 0; d < ndof; ++d) de_ptr[d + 1] += de_ptr[d];
    std::vector<double> darea(ndof, 0.0);
    {
        std::vector<int> cur(de_ptr.begin(), de_ptr.end() - 1);
        for (int e = 0; e < E; ++e)
            for (int a = 0; a < 3; ++a) {
                const int d = edof[3 * e + a];
                de_el[cur[d]++] = 3 * e + a;
                darea[d] += area[e];
            }
    }
    // matrix pattern, mass and stiffness matrices, and per-entry contribution lists
    std::vector<std::map<int, std::vector<int>>> rows(ndof);
    for (int e = 0; e < E; ++e)
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b) rows[edof[3 * e + a]][edof[3 * e + b]].push_back(9 * e + 3 * a + b);
    std::vector<int> row(ndof + 1, 0), col, cptr(1, 0), cel;
    std::vector<double> Mval, Kval, Kdiag(ndof, 0.0);
    for (int i = 0; i < ndof; ++i) {
        for (const auto& kv : rows[i]) {
            col.push_back(kv.first);
            double m = 0.0, kk = 0.0;
            for (int c : kv.second) {
                const int e = c / 9, a = (c / 3) % 3, b = c % 3;
                const double* g = &grad[6 * (size_t)e];
                m += area[e] / 12.0 * (a == b ? 2.0 : 1.0);
                kk += area[e] * (g[2 * a] * g[2 * b] + g[2 * a + 1] * g[2 * b + 1]);
                cel.push_back(c);
            }
            cptr.push_back((int)cel.size());
            Mval.push_back(m);
            Kval.push_back(kk);
            if (kv.first == i) Kdiag[i] = kk;
        }
        row[i + 1] = (int)col.size();
    }
    // wall DOFs with the averaged inward unit normal (left of each CCW boundary edge)
    std::vector<unsigned char> wall(ndof, 0);
    std::vector<double> normal(2 * (size_t)ndof, 0.0);
    for (int e = 0; e < E; ++e)
        for (int k = 0; k < 3; ++k) {
            const int t = tag[3 * e + k];
            if (t != LPDF_EDGE_WALL && t != LPDF_EDGE_MOVING_WALL) continue;
            const int a = tri[3 * e + k], b = tri[3 * e + (k + 1) % 3];
            const double tx = node_xy[2 * b] - node_xy[2 * a], ty = node_xy[2 * b + 1] - node_xy[2 * a + 1];
            const double len = std::hypot(tx, ty);
            for (int v : {a, b}) {
                const int d = dof[v];
                wall[d] = 1;
                normal[2 * d] += -ty / len;
                normal[2 * d + 1] += tx / len;
            }
        }
    // wall edges grouped by component (components own contiguous element ranges, in order)
    const int n_comp = node_comp.empty() ? 1 : *std::max_element(node_comp.begin(), node_comp.end()) + 1;
    std::vector<double> seg;
    std::vector<int> segn, seg_off(n_comp + 1, 0);
    for (int e = 0; e < E; ++e)
        for (int k = 0; k < 3; ++k) {
            const int t = tag[3 * e + k];
            if (t != LPDF_EDGE_WALL && t != LPDF_EDGE_MOVING_WALL) continue;
            const int a = tri[3 * e + k], b = tri[3 * e + (k + 1) % 3];
            seg.insert(seg.end(), {node_xy[2 * a], node_xy[2 * a + 1], node_xy[2 * b], node_xy[2 * b + 1]});
            segn.insert(segn.end(), {a, b});
            ++seg_off[(node_comp.empty() ? 0 : node_comp[a]) + 1];
        }
    for (int c = 0; c < n_comp; ++c) seg_off[c + 1] += seg_off[c];
    std::vector<int> ncomp_v(N, 0);
    for (int i = 0; i < N && !node_comp.empty(); ++i) ncomp_v[i] = node_comp[i];
    const std::vector<double> xy(node_xy, node_xy + 2 * (size_t)N);
    for (int d = 0; d < ndof; ++d)
        if (wall[d]) {
            const double l = std::hypot(normal[2 * d], normal[2 * d + 1]);
            normal[2 * d] /= l;
            normal[2 * d + 1] /= l;
        }
    std::vector<double> iarea(ndof);
    for (int d = 0; d < ndof; ++d) iarea[d] = 1.0 / darea[d];
    Fem* F = new Fem();
    F->ndof = ndof;
    F->nnz = (int)col.size();
    F->E = E;
    F->N = N;
    F->nseg = (int)(seg.size() / 4);
    F->n_comp = n_comp;
    F->period = period;
    for (int i = 0; i < ndof; ++i) {
        double total = 0.0;
        for (int t = row[i]; t < row[i + 1]; ++t) total += std::fabs(Kval[t]);
        F->lmaxK = std::max(F->lmaxK, total / Kdiag[i]);
    }
    // cg_kernel's partition (one CTA per SM): every CTA's rows of others that its rows refer to, and the
    // columns as indices into (its own rows, those)
    F->cg_ctas = sm_count();
    const int parts = std::max(1, std::min(F->cg_ctas, (ndof + 31) / 32));
    std::vector<int> halo_ptr(parts + 1, 0), halo, lcol(col.size()), local(ndof, -1);
    for (int b = 0; b < parts; ++b) {
        const int lo = (int)((int64_t)ndof * b / parts), hi = (int)((int64_t)ndof * (b + 1) / parts);
        const size_t h0 = halo.size();
        for (int t = row[lo]; t < row[hi]; ++t)
            if ((col[t] < lo || col[t] >= hi) && local[col[t]] != b) {
                local[col[t]] = b;
                halo.push_back(col[t]);
            }
        std::sort(halo.begin() + h0, halo.end());
        for (int t = row[lo]; t < row[hi]; ++t)
            lcol[t] = col[t] >= lo && col[t] < hi
                          ? col[t] - lo
                          : hi - lo + (int)(std::lower_bound(halo.begin() + h0, halo.end(), col[t]) - halo.begin() - h0);
        halo_ptr[b + 1] = (int)halo.size();
        F->max_halo = std::max(F->max_halo, halo_ptr[b + 1] - halo_ptr[b]);
        F->max_slice = std::max(F->max_slice, row[hi] - row[lo]);
    }
    if (halo.empty()) halo.push_back(0);
    for (int i = 0; i < ndof; ++i) F->max_deg = std::max(F->max_deg, row[i + 1] - row[i]);
    if (seg.empty()) {
        seg.assign(4, 0.0);
        segn.assign(2, 0);
    }
    cudaError_t e = cudaSuccess;
    if ((e = upload(&F->dof, dof)) || (e = upload(&F->dof_node, dof_node)) || (e = upload(&F->edof, edof)) ||
        (e = upload(&F->area, area)) || (e = upload(&F->grad, grad)) || (e = upload(&F->de_ptr, de_ptr)) ||
        (e = upload(&F->de_el, de_el)) || (e = upload(&F->iarea, iarea)) || (e = upload(&F->row, row)) ||
        (e = upload(&F->col, col)) || (e = upload(&F->lcol, lcol)) || (e = upload(&F->halo_ptr, halo_ptr)) ||
        (e = upload(&F->halo, halo)) || (e = upload(&F->cptr, cptr)) || (e = upload(&F->cel, cel)) ||
        (e = upload(&F->Mval, Mval)) || (e = upload(&F->Kval, Kval)) || (e = upload(&F->Kdiag, Kdiag)) || (e = upload(&F->wall, wall)) ||
        (e = upload(&F->normal, normal)) || (e = upload(&F->xy, xy)) || (e = upload(&F->seg, seg)) ||
        (e = upload(&F->segn, segn)) || (e = upload(&F->seg_off, seg_off)) || (e = upload(&F->ncomp, ncomp_v)) || (e = cudaMalloc((void**)&F->wdist, sizeof(double) * std::max(1, N))) ||
        (e = cudaMalloc((void**)&F->wseg, sizeof(int) * std::max(1, N))) ||
        (e = cudaMalloc((void**)&F->wt, sizeof(double) * std::max(1, N))) ||
        (e = cudaMalloc((void**)&F->Aval, sizeof(double) * std::max(1, F->nnz))) ||
        (e = cudaMalloc((void**)&F->work, sizeof(double) * (Fem::kWorkPerDof * (size_t)ndof + 16 * (size_t)E))) ||
        (e = cudaMalloc((void**)&F->part, sizeof(double) * Fem::kDotBlocks)) ||
        (e = cudaMalloc(&F->cg_slots, sizeof(ulonglong2) * cg_slot_words(F->cg_ctas))) ||
        (e = cudaMemset(F->cg_slots, 0, sizeof(ulonglong2) * cg_slot_words(F->cg_ctas))) ||
        (e = cudaMalloc((void**)&F->cg_z, sizeof(ulonglong2) * kCgComps * ((size_t)ndof + 255))) ||
        (e = cudaMemset(F->cg_z, 0, sizeof(ulonglong2) * kCgComps * ((size_t)ndof + 255))) ||
        (e = cudaMalloc((void**)&F->cg_zp, sizeof(ulonglong2) * 2 * kCgComps * (size_t)ndof)) ||
        (e = cudaMemset(F->cg_zp, 0, sizeof(ulonglong2) * 2 * kCgComps * (size_t)ndof)) ||
        (e = cudaMalloc((void**)&F->lmax, sizeof(double))) ||
        (e = cudaMalloc((void**)&F->cg_out, sizeof(int) * kCgOut)) ||
        (e = cudaMallocHost((void**)&F->cg_host, sizeof(int) * kCgOut)) || (e = cg_configure())) {
        fem_free(F);
        return e;
    }
    *out = F;
    return cudaSuccess;
}

void fem_free(Fem* F)
{
    if (!F) return;
    void* ps[] = {F->dof, F->dof_node, F->edof, F->area, F->grad, F->de_ptr, F->de_el, F->iarea, F->row, F->col, F->lcol, F->halo_ptr, F->halo,
                  F->cptr, F->cel, F->Mval, F->Kval, F->Kdiag, F->Aval, F->wall, F->normal, F->work, F->part, F->cg_slots, F->cg_z, F->cg_zp, F->lmax, F->cg_out,
                  F->xy, F->seg, F->segn, F->seg_off, F->ncomp, F->wdist, F->wseg, F->wt};
    for (void* p : ps) cudaFree(p);
    cudaFreeHost(F->cg_host);
    delete F;
}

namespace {

// One cooperative launch of the CG on the systems that `a` names (its matrices, right-hand sides,
// starts, component counts and scratch set). At least 32 rows per CTA: fewer CTAs have fewer
// partial sums to exchange. The line between the kernels lies where the small one's warps poll two
// words per lane; it needs rows of at most kCgDeg entries.
cudaError_t launch_cg(Fem& F, CgArgs& a, cudaStream_t st)
{
    const int n = F.ndof;
    a.n = n;
    a.row = F.row;
    a.col = F.col;
    a.wall = F.wall;
    a.slots = static_cast<ulonglong2*>(F.cg_slots);
    a.out = F.cg_out;
    a.polls = F.cg_polls;
    a.quit = F.cg_quit;
    a.epoch = F.cg_epoch;
    F.cg_epoch += (unsigned long long)a.maxit + 4ull;
    const cudaError_t e = cudaMemsetAsync(F.cg_out, 0, sizeof(int) * kCgOut, st);
    if (e != cudaSuccess) return e;
    void* args[] = {&a};
    if (n <= kCgSmallRows && F.max_deg <= kCgDeg)
        return cudaLaunchCooperativeKernel((const void*)cg_small_kernel, dim3(8 * ((n + 255) / 256) * a.nc), dim3(32),
                                           args, 0, st);
    const int G = std::max(1, std::min(F.cg_ctas, (n + 31) / 32));
    const int rows = (n + G - 1) / G;
    a.wpc = std::min((kCgMaxThreads / 32 - kCgTasks) / a.nc, (rows + 31) / 32);
    const int slice = F.max_slice;
    const bool one = rows <= 32 * a.wpc;
    const int systems = (a.nv0 > 0) + (a.nc > a.nv0);
    a.width = rows + F.max_halo;
    size_t bytes = slice * (sizeof(int) + sizeof(double) * systems);
    const size_t poly = bytes + a.nc * (size_t)a.width * 2 * sizeof(double) + sizeof(int) * (size_t)F.max_halo;
    const bool smem = one ? poly <= kCgPolySmemMax : bytes <= kCgSmemMax;
    if (one) bytes = poly;
    if (one && smem) {
        const double lo = 1.0 / kChebRatio, sigma = (1.0 + lo) / (1.0 - lo);
        a.cheb[0] = 2.0 / (1.0 + lo);
        double rho = 1.0 / sigma;
        for (int k = 0; k < kCheb; ++k) {
            const double next = 1.0 / (2.0 * sigma - rho);
            a.cheb[1 + 2 * k] = next * rho;
            a.cheb[2 + 2 * k] = 4.0 * next / (1.0 - lo);
            rho = next;
        }
        a.epochp = F.cg_epochp;
        F.cg_epochp += (unsigned long long)kCheb * ((unsigned long long)a.maxit + 2ull);
        a.zp = F.cg_zp;
        a.lcol = F.lcol;
        a.halo_ptr = F.halo_ptr;
        a.halo = F.halo;
    }
    a.slice = smem ? slice : 0;
    const void* fn = one ? (smem ? (const void*)cg_kernel<true, true> : (const void*)cg_kernel<true, false>)
                         : (smem ? (const void*)cg_kernel<false, true> : (const void*)cg_kernel<false, false>);
    return cudaLaunchCooperativeKernel(fn, dim3(G), dim3(32 * (a.nc * a.wpc + kCgTasks)), args, smem ? bytes : 0, st);
}

}  // namespace

cudaError_t node_fields_solve(Fem& F, const double* stats, const lpdf_params& P, float* out, double tol,
                              int maxit, int* iters, cudaStream_t st, const float* surr, const float* surr_norm)
{
    const int ns = P.ns;
    const size_t n = F.ndof;
    const int nq = nquant(ns);
    const int nfp = nfields_padded(ns);
    double* w = F.work;
    double* U = w;      w += 3 * n;
    double* R = w;      w += 6 * n;
    double* om = w;     w += n;
    double* phi = w;    w += (size_t)kMaxNS * n;
    double* k = w;      w += n;
    double* eps = w;    w += n;
    double* gU = w;     w += 6 * n;
    double* lapU = w;   w += 3 * n;
    double* gp = w;     w += 2 * n;
    double* wp = w;     w += 4 * n;
    double* p = w;      w += n;
    double* diag = w;   w += n;
    double* rhs = w;    w += 5 * n;       // the relaxation's four, the pressure's
    double* tmp = w;    w += 4 * n;
    double* L2 = w;     w += n;
    double* cgs = w;    w += 20 * n;      // scratch of the CG
    double* xref = w;   w += 5 * n;       // the zero-interior start (reference of the test)
    double* wp_prev = w; w += 4 * n;      // previous solutions (warm start)
    double* p_prev = w; w += n;
    double* ew = F.work + Fem::kWorkPerDof * n;   // element scratch, 16 per element
    const unsigned gd = blocks((int64_t)n), ge = blocks(F.E);
    iters[0] = iters[1] = 0;
    const bool relax = P.gmodel == 0 && !surr, press = P.pressure_solve != 0;
    dof_stats_kernel<<<gd, 256, 0, st>>>(F, stats, nq, ns, P.CL, P.Ceta * std::pow(P.nu, 0.75), U, R, om, phi, k, eps,
                                         relax ? L2 : nullptr);
    // recovered gradients of the mean velocity, then their recovered divergences
    elem_grad_kernel<<<ge, 256, 0, st>>>(F, U, 3, 3, ew);
    recover_kernel<<<blocks(6 * (int64_t)n), 256, 0, st>>>(F, ew, 6, gU, 6);
    elem_div_kernel<<<blocks(3 * (int64_t)F.E), 256, 0, st>>>(F, gU, ew);
    recover_kernel<<<blocks(3 * (int64_t)n), 256, 0, st>>>(F, ew, 3, lapU, 3);
    CgArgs a{};
    a.tol = tol;
    a.maxit = maxit;
    a.z = F.cg_z;
    a.lmax0 = F.lmax;
    a.lmax1 = F.lmaxK;
    a.state = cgs;
    if (relax) {
        elem_L2_kernel<<<ge, 256, 0, st>>>(F, L2, ew);
        const cudaError_t e = cudaMemsetAsync(F.lmax, 0, sizeof(double), st);
        if (e != cudaSuccess) return e;
        assemble_kernel<<<gd, 256, 0, st>>>(F, ew, F.Aval, diag, F.lmax);
        const bool warm = P.cg_warm_start && F.has_wp;
        er_setup_kernel<<<gd, 256, 0, st>>>(F, eps, P.C0, tmp, wp, warm ? wp_prev : nullptr, xref);
        spmv_kernel<<<gd, 256, 0, st>>>(F, F.Mval, tmp, rhs);     // b = M wp^h
        a.A0 = F.Aval;
        a.d0 = diag;
        a.b0 = rhs;
        a.x0 = wp;
        a.ref0 = xref;
        a.mask0 = 1;
        a.nv0 = 4;
    }
    a.nc = a.nv0;
    if (press) {
        pressure_T_kernel<<<gd, 256, 0, st>>>(F, U, R, tmp);
        elem_grad_kernel<<<ge, 256, 0, st>>>(F, tmp, 4, 4, ew);
        pressure_rhs_kernel<<<gd, 256, 0, st>>>(F, ew, rhs + 4 * n);
        // consistent singular system (the right-hand side sums to zero): CG stays in the range up
        // to rounding; the constant is removed afterwards. Reference start: zero.
        const bool warm = P.cg_warm_start && F.has_p;
        cudaError_t e = warm ? cudaMemcpyAsync(p, p_prev, sizeof(double) * n, cudaMemcpyDeviceToDevice, st)
                             : cudaMemsetAsync(p, 0, sizeof(double) * n, st);
        if (e == cudaSuccess && warm) e = cudaMemsetAsync(xref + 4 * n, 0, sizeof(double) * n, st);
        if (e != cudaSuccess) return e;
        a.A1 = F.Kval;
        a.d1 = F.Kdiag;
        a.b1 = rhs + 4 * n;
        a.x1 = p;
        a.ref1 = warm ? xref + 4 * n : nullptr;
        ++a.nc;
    }
    if (a.nc > 0) {
        const cudaError_t e = launch_cg(F, a, st);
        if (e != cudaSuccess) return e;
    }
    if (press) {
        const int nb = (int)std::min<unsigned>(Fem::kDotBlocks, blocks((int64_t)n, kDotThreads));   // fixed order
        sum_kernel<<<nb, kDotThreads, 0, st>>>(p, (int)n, F.part);
        subtract_mean_kernel<<<gd, 256, 0, st>>>((int)n, F.part, nb, p);
        elem_grad_kernel<<<ge, 256, 0, st>>>(F, p, 1, 1, ew);
        recover_kernel<<<blocks(2 * (int64_t)n), 256, 0, st>>>(F, ew, 2, gp, 2);
    } else {
        const cudaError_t e = cudaMemsetAsync(gp, 0, sizeof(double) * 2 * n, st);
        if (e != cudaSuccess) return e;
    }
    fields_kernel<<<blocks(F.N), 256, 0, st>>>(F, ns, nfp, U, R, om, phi, k, eps, gU, lapU, gp, wp, P.gmodel, P.C0,
                                               P.Comega1, P.Comega2, P.dpdx0, P.dpdy0, surr, surr_norm,
                                               a.nc > 0 ? F.cg_out : nullptr, relax + press, out);
    if (a.nc == 0) return cudaGetLastError();
    // everything is enqueued: the one synchronisation reads how the CGs ended
    const int n4 = relax ? 4 * (int)n : 0, n1 = press ? (int)n : 0;
    keep_solution_kernel<<<blocks(std::max(n4, n1)), 256, 0, st>>>(F.cg_out, relax + press, n4, wp, wp_prev, n1, p, p_prev);
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess)
        e = cudaMemcpyAsync(F.cg_host, F.cg_out, sizeof(int) * kCgOut, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return e;
    if (F.cg_host[kCgError]) return cudaErrorLaunchTimeout;   // a bounded wait of the CG kernel gave up
    iters[0] = F.cg_host[kCgIts0];
    iters[1] = F.cg_host[kCgIts1];
    if (F.cg_host[kCgOk] != relax + press) return cudaErrorNotReady;
    F.has_wp = F.has_wp || relax;
    F.has_p = F.has_p || press;
    return cudaSuccess;
}

cudaError_t surrogate_features(Fem& F, const double* stats, int ns, const float* fields, double C0, float* feat,
                               float* tgt, cudaStream_t st)
{
    if (!F.has_wdist) {
        wall_distance_kernel<<<blocks(F.N), 256, 0, st>>>(F.N, F.xy, F.seg, F.seg_off, F.ncomp, F.period, F.wdist,
                                                          F.wseg, F.wt);
        F.has_wdist = true;
    }
    features_kernel<<<blocks(F.N), 256, 0, st>>>(F, stats, nquant(ns), fields, nfields_padded(ns), C0, feat,
                                                 fields ? tgt : nullptr);
    return cudaGetLastError();
}

cudaError_t fields_compare(const float* a, const float* b, int n_nodes, int nfp, double* out2, cudaStream_t st)
{
    fields_compare_kernel<<<1, 1024, 0, st>>>(a, b, n_nodes, nfp, out2);
    return cudaGetLastError();
}

}  // namespace lpdf
