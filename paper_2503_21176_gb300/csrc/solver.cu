// Regular QEq by GMRES and regular Born-Oppenheimer MD (Sec. 3.4, Sec. 4.1).
//
// The bordered system of Eq. linear_qeq,
//     [diag(u) + Phi   1] [q     ]   [-chi ]
//     [1^T             0] [lambda] = [Q_tot],
// is solved by restarted GMRES with a right Jacobi preconditioner
// M = diag(u_i + g_i, 1), where g_i = k_e sqrt(2/pi) / sigma_i is the Gaussian
// self-energy when that term is on (the dominant part of Phi_ii), else 0.
// Right preconditioning keeps the monitored residual the true one,
// ||b - A z|| / ||b||.  That is the paper's tolerance.  Each Arnoldi vector
// costs one potential-only Coulomb apply.  Vectors have N + 1 entries, the
// last one being lambda.  Orthogonalisation is classical Gram-Schmidt done
// twice in three kernels; an iteration is five launches beside its apply (sums
// finish in the last block of their kernel, scaling runs with the preconditioner,
// a subtraction with the dots or the norm that follow it).  The
// (m + 1) x m Hessenberg least-squares problem is reduced by Givens rotations
// on the host from one small device-to-host copy per iteration.
//
// The regular BO-MD step: velocity-Verlet half kick and drift, a neighbour
// rebuild when due, a solve warm-started from the previous charges, one apply
// with the field for F = q o E (+ short range), and the second half kick.  The
// potential energy is sum q chi + 1/2 sum u q^2 + 1/2 q.Phi q (+ short range)
// at the approximate charges.
#include <cmath>
#include <vector>

#include "internal.cuh"

namespace qeq {

namespace {

constexpr int kMaxDots = kMaxGmresRestart;  // Gram-Schmidt against at most this many vectors

// y = A x for x = [xq; xl]:  y_q = u o xq + Phi xq + xl,  y_l = sum xq.
// phi holds Phi xq; the last block to finish writes y_l.
__global__ void k_bordered_apply(int n, const double *__restrict__ u, const double *__restrict__ phi,
                                 const double *__restrict__ x, double *__restrict__ y,
                                 double *__restrict__ part, unsigned int *__restrict__ ticket) {
    const double xl = x[n];
    double s = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        y[i] = u[i] * x[i] + phi[i] + xl;
        s += x[i];
    }
    double vals[1] = {s};
    block_sum<1>(vals);
    if (threadIdx.x == 0) part[blockIdx.x] = vals[0];
    finalize_last_block<1>(part, y + n, ticket);
}

// v = a x over n + 1 entries, and z = M^{-1} v (q part times dinv, lambda unchanged);
// v may be x.
__global__ void k_scale_precond(int n, double a, const double *x, double *v,
                                const double *__restrict__ dinv, double *__restrict__ z) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) {
        const double t = a * x[i];
        v[i] = t;
        z[i] = i < n ? t * dinv[i] : t;
    }
}

// Partials of <V_k, w>, k < nv, over n1 entries (slot k): eight vectors a pass, so w is
// read once for them and their sums fold together.
__device__ __forceinline__ void dots(int n1, int nv, const double *__restrict__ V, const double *w,
                                     double *__restrict__ part) {
    for (int k0 = 0; k0 < nv; k0 += 8) {
        double s[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
        for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n1; i += gridDim.x * blockDim.x) {
            const double wi = w[i];
#pragma unroll
            for (int u = 0; u < 8; ++u)
                if (k0 + u < nv) s[u] = fma(V[(size_t)(k0 + u) * n1 + i], wi, s[u]);
        }
        block_sum<8>(s);
        if (threadIdx.x == 0)
            for (int u = 0; u < 8 && k0 + u < nv; ++u) part[(size_t)(k0 + u) * kRedBlocks + blockIdx.x] = s[u];
    }
}

// The last block to arrive sums nslots slots' partials in a fixed order, one warp a slot.
__device__ __forceinline__ void finalize_slots(int nslots, const double *part, double *out,
                                               unsigned int *ticket) {
    __shared__ bool is_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) is_last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!is_last) return;
    __threadfence();
    const int lane = threadIdx.x & 31;
    for (int k = threadIdx.x >> 5; k < nslots; k += kThreads / 32) {
        double t = 0.0;
        for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(part + (size_t)k * kRedBlocks + b);
        t = warp_sum(t);
        if (lane == 0) out[k] = t;
    }
    if (threadIdx.x == 0) *ticket = 0u;
}

// h_k = <V_k, w>, k < nv
__global__ void k_multi_dot(int n1, int nv, const double *__restrict__ V, const double *__restrict__ w,
                            double *__restrict__ part, double *__restrict__ h,
                            unsigned int *__restrict__ ticket) {
    dots(n1, nv, V, w, part);
    finalize_slots(nv, part, h, ticket);
}

// w -= sum_k h_k V_k, then (again) h2_k = <V_k, w> or (norm) h2_0 = <w, w>: each thread
// owns its entries of w, so the subtraction and the next dots need one launch.
__global__ void k_subtract_dot(int n1, int nv, const double *__restrict__ V, const double *__restrict__ h,
                               double *w, bool norm, double *__restrict__ part, double *__restrict__ h2,
                               unsigned int *__restrict__ ticket) {
    __shared__ double hs[kMaxDots];
    for (int k = threadIdx.x; k < nv; k += blockDim.x) hs[k] = h[k];
    __syncthreads();
    double n2 = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n1; i += gridDim.x * blockDim.x) {
        double s = w[i];
        for (int k = 0; k < nv; ++k) s -= hs[k] * V[(size_t)k * n1 + i];
        w[i] = s;
        n2 = fma(s, s, n2);
    }
    if (norm) {
        double vals[1] = {n2};
        block_sum<1>(vals);
        if (threadIdx.x == 0) part[blockIdx.x] = vals[0];
        finalize_last_block<1>(part, h2, ticket);
    } else {
        dots(n1, nv, V, w, part);
        finalize_slots(nv, part, h2, ticket);
    }
}

// r = b - Az with b = [-chi; q_tot] (Az null: b itself), and |r|^2; r may be Az
__global__ void k_residual(int n, double q_tot, const double *__restrict__ chi, const double *Az, double *r,
                           double *__restrict__ part, double *__restrict__ r2,
                           unsigned int *__restrict__ ticket) {
    double s = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) {
        const double ri = (i < n ? -chi[i] : q_tot) - (Az ? Az[i] : 0.0);
        r[i] = ri;
        s = fma(ri, ri, s);
    }
    double vals[1] = {s};
    block_sum<1>(vals);
    if (threadIdx.x == 0) part[blockIdx.x] = vals[0];
    finalize_last_block<1>(part, r2, ticket);
}

// z += M^{-1} (sum_k y_k V_k)
__global__ void k_update_solution(int n, int nv, const double *__restrict__ V,
                                  const double *__restrict__ y, const double *__restrict__ dinv,
                                  double *__restrict__ z) {
    const int n1 = n + 1;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += gridDim.x * blockDim.x) {
        double s = 0.0;
        for (int k = 0; k < nv; ++k) s += y[k] * V[(size_t)k * n1 + i];
        z[i] += i < n ? s * dinv[i] : s;
    }
}

__global__ void k_jacobi(int n, const double *__restrict__ u, const double *__restrict__ sigma,
                         double gauss_coef, double *__restrict__ dinv) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double d = u[i];
        if (gauss_coef != 0.0 && sigma[i] > 0.0) d += gauss_coef / sigma[i];
        dinv[i] = 1.0 / d;
    }
}

// q part of z into q, and the energy partials: sum q chi, sum u q^2 / 2, sum q v / 2, sum q
__global__ void k_bo_energy_part(int n, const double *__restrict__ q, const double *__restrict__ chi,
                                 const double *__restrict__ u, const double *__restrict__ v,
                                 double *__restrict__ part) {
    double a[4] = {0, 0, 0, 0};
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        a[0] += q[i] * chi[i];
        a[1] += 0.5 * u[i] * q[i] * q[i];
        a[2] += 0.5 * q[i] * v[i];
        a[3] += q[i];
    }
    block_sum<4>(a);
    if (threadIdx.x == 0)
        for (int k = 0; k < 4; ++k) part[(size_t)k * kRedBlocks + blockIdx.x] = a[k];
}

__global__ void k_bo_forces(int n, const double *__restrict__ q, const double *__restrict__ E,
                            const double *__restrict__ Fs, double *__restrict__ F) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            double f = q[i] * E[3 * (size_t)i + d];
            if (Fs) f += Fs[3 * (size_t)i + d];
            F[3 * (size_t)i + d] = f;
        }
}

// energies: 1 potential (BO energy + short), 3 short, 4 lambda, 5 sum q, 6 rel residual, 7 applies
__global__ void k_bo_energies(const double *__restrict__ sums, const double *__restrict__ e_short2,
                              double lambda, double relres, double applies,
                              double *__restrict__ energies) {
    const double es = e_short2[0] + e_short2[1];
    energies[1] = sums[0] + sums[1] + sums[2] + es;
    energies[3] = es;
    energies[4] = lambda;
    energies[5] = sums[3];
    energies[6] = relres;
    energies[7] = applies;
}

}  // namespace

int short_range_forces(qeq_ctx *ctx, const double *R, const double *mass, double *F_short,
                       double *e_slot, cudaStream_t s);

int solver_alloc(qeq_ctx *ctx, int restart) {
    if (ctx->gm_restart >= restart && ctx->gmV) return QEQ_OK;
    dev_free(ctx, ctx->gmV);
    dev_free(ctx, ctx->gmW);
    dev_free(ctx, ctx->gmZ);
    dev_free(ctx, ctx->gmDinv);
    dev_free(ctx, ctx->gmH);
    ctx->gmV = ctx->gmW = ctx->gmZ = ctx->gmDinv = ctx->gmH = nullptr;
    const size_t n1 = (size_t)ctx->n + 1;
    int rc = dev_alloc(ctx, (void **)&ctx->gmV, sizeof(double) * n1 * (restart + 1));
    if (!rc) rc = dev_alloc(ctx, (void **)&ctx->gmW, sizeof(double) * n1 * 2);
    if (!rc) rc = dev_alloc(ctx, (void **)&ctx->gmZ, sizeof(double) * n1);
    if (!rc) rc = dev_alloc(ctx, (void **)&ctx->gmDinv, sizeof(double) * n1);
    if (!rc) rc = dev_alloc(ctx, (void **)&ctx->gmH, sizeof(double) * (kMaxDots + 4) * 2);
    if (rc) return rc;
    ctx->gm_restart = restart;
    return QEQ_OK;
}

void solver_free(qeq_ctx *ctx) {
    dev_free(ctx, ctx->gmV);
    dev_free(ctx, ctx->gmW);
    dev_free(ctx, ctx->gmZ);
    dev_free(ctx, ctx->gmDinv);
    dev_free(ctx, ctx->gmH);
    dev_free(ctx, ctx->gmSol);
}

namespace {

// Orthogonalise w against V_0..V_{nv-1}, classical Gram-Schmidt twice: three launches
// (dots; subtract and dots again; subtract and norm).  Small vectors are bound by the
// launches: 20,000 atoms in FP64 took 17.3 ms with twelve launches an iteration beside
// the apply, 14.2 ms with five.  Long ones are bound by reading V four times.
// On return h[k] is the sum of both passes' coefficients and norm = |w|.
int cgs2(qeq_ctx *ctx, int n1, int nv, double *w, std::vector<double> &h, double &norm,
         cudaStream_t s) {
    double *part = ctx->part;
    double *dh = ctx->gmH;  // pass 1 at [0, nv), pass 2 at [kMaxDots + 2, ...), |w|^2 at the end
    const int off2 = kMaxDots + 2;
    const int G = ctx->atom_grid;
    k_multi_dot<<<G, kThreads, 0, s>>>(n1, nv, ctx->gmV, w, part, dh, ctx->ticket);
    k_subtract_dot<<<G, kThreads, 0, s>>>(n1, nv, ctx->gmV, dh, w, false, part, dh + off2, ctx->ticket);
    k_subtract_dot<<<G, kThreads, 0, s>>>(n1, nv, ctx->gmV, dh + off2, w, true, part, dh + 2 * off2,
                                          ctx->ticket);
    ctx->launches += 3;
    double hb[2 * (kMaxDots + 2) + 1];
    cudaError_t e = cudaMemcpyAsync(hb, dh, sizeof(hb), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    int rc = cuda_check(ctx, e, "gmres orthogonalise");
    if (rc) return rc;
    h.assign(nv, 0.0);
    for (int k = 0; k < nv; ++k) h[k] = hb[k] + hb[off2 + k];
    norm = std::sqrt(std::max(0.0, hb[2 * off2]));
    return QEQ_OK;
}

// y = A x  (one potential-only Coulomb apply)
int bordered_apply(qeq_ctx *ctx, const double *R, const double *u, const double *sigma,
                   const double *x, double *y, cudaStream_t s, bool same_R) {
    const int n = (int)ctx->n;
    int rc = coulomb_apply_impl(ctx, R, x, sigma, ctx->phi, nullptr, nullptr, nullptr, false, s,
                                same_R, true);
    if (rc) return rc;
    k_bordered_apply<<<ctx->atom_grid, kThreads, 0, s>>>(n, u, ctx->phi, x, y, ctx->part, ctx->ticket);
    ctx->launches++;
    return QEQ_OK;
}

// r = b - Az (Az null: b) and its norm on the host
double residual_norm(qeq_ctx *ctx, const double *chi, const double *Az, double *r, cudaStream_t s, int *rc) {
    k_residual<<<ctx->atom_grid, kThreads, 0, s>>>((int)ctx->n, ctx->p.q_tot, chi, Az, r, ctx->part, ctx->gmH,
                                                   ctx->ticket);
    ctx->launches++;
    double v = 0.0;
    cudaError_t e = cudaMemcpyAsync(&v, ctx->gmH, sizeof(double), cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    *rc = cuda_check(ctx, e, "gmres norm");
    return std::sqrt(std::max(0.0, v));
}

}  // namespace

// Solve the bordered QEq system; z (device, N + 1) holds the initial guess
// [q; lambda] on entry and the solution on exit.
int gmres_solve(qeq_ctx *ctx, const double *R, const double *chi, const double *u,
                const double *sigma, double *z, double tol, int max_iter, int restart,
                bool final_check, qeq_solve_info *info, cudaStream_t s) {
    const int n = (int)ctx->n;
    const int n1 = n + 1;
    restart = std::max(1, std::min(restart, kMaxDots));
    int rc = solver_alloc(ctx, restart);
    if (rc) return rc;
    pair_reserve(ctx, s);  // every iteration's apply is at these positions
    const qeq_params &p = ctx->p;
    k_jacobi<<<ctx->red_grid, kThreads, 0, s>>>(n, u, sigma, p.gaussian_self ? p.k_e * kSqrtTwoOverPi : 0.0,
                                             ctx->gmDinv);
    ctx->launches++;
    double *w = ctx->gmW;       // A z, then the residual / Arnoldi work vector
    double *bvec = ctx->gmW + n1;
    // |b| with b = [-chi; q_tot]
    double bnorm = residual_norm(ctx, chi, nullptr, bvec, s, &rc);
    if (rc) return rc;
    if (!(bnorm > 0.0)) bnorm = 1.0;
    int iters = 0, applies = 0;
    double relres = 1.0;
    std::vector<double> H((size_t)(restart + 1) * restart), cs(restart), sn(restart), g(restart + 1), h;
    while (true) {
        // r = b - A z
        rc = bordered_apply(ctx, R, u, sigma, z, w, s, applies > 0);
        if (rc) return rc;
        ++applies;
        const double beta = residual_norm(ctx, chi, w, w, s, &rc);
        if (rc) return rc;
        relres = beta / bnorm;
        if (relres <= tol || iters >= max_iter || !(beta > 0.0)) break;
        std::fill(g.begin(), g.end(), 0.0);
        g[0] = beta;
        double scale = 1.0 / beta;  // of the vector that becomes V_j, still unscaled in from
        const double *from = w;
        int j = 0;
        for (; j < restart && iters < max_iter; ++j) {
            double *vj = ctx->gmV + (size_t)j * n1;
            double *vnext = ctx->gmV + (size_t)(j + 1) * n1;
            k_scale_precond<<<ctx->atom_grid, kThreads, 0, s>>>(n, scale, from, vj, ctx->gmDinv, ctx->gmZ);
            ctx->launches++;
            rc = bordered_apply(ctx, R, u, sigma, ctx->gmZ, vnext, s, applies > 0);
            if (rc) return rc;
            ++applies;
            ++iters;
            double hn;
            rc = cgs2(ctx, n1, j + 1, vnext, h, hn, s);
            if (rc) return rc;
            for (int k = 0; k <= j; ++k) H[(size_t)k * restart + j] = h[k];
            H[(size_t)(j + 1) * restart + j] = hn;
            scale = hn > 0.0 ? 1.0 / hn : 1.0;
            from = vnext;
            // apply the previous rotations to column j, then a new one
            for (int k = 0; k < j; ++k) {
                const double a = H[(size_t)k * restart + j], b = H[(size_t)(k + 1) * restart + j];
                H[(size_t)k * restart + j] = cs[k] * a + sn[k] * b;
                H[(size_t)(k + 1) * restart + j] = -sn[k] * a + cs[k] * b;
            }
            const double a = H[(size_t)j * restart + j], b = H[(size_t)(j + 1) * restart + j];
            const double rr = std::hypot(a, b);
            cs[j] = rr > 0.0 ? a / rr : 1.0;
            sn[j] = rr > 0.0 ? b / rr : 0.0;
            H[(size_t)j * restart + j] = rr;
            H[(size_t)(j + 1) * restart + j] = 0.0;
            g[j + 1] = -sn[j] * g[j];
            g[j] = cs[j] * g[j];
            relres = std::fabs(g[j + 1]) / bnorm;
            if (relres <= tol || !(hn > 0.0)) {
                ++j;
                break;
            }
        }
        // y = H^{-1} g (upper triangular j x j), z += M^{-1} V y
        std::vector<double> y(j, 0.0);
        for (int r = j - 1; r >= 0; --r) {
            double acc = g[r];
            for (int c = r + 1; c < j; ++c) acc -= H[(size_t)r * restart + c] * y[c];
            const double d = H[(size_t)r * restart + r];
            y[r] = d != 0.0 ? acc / d : 0.0;
        }
        cudaError_t e = cudaMemcpyAsync(ctx->gmH, y.data(), sizeof(double) * std::max(1, j),
                                        cudaMemcpyHostToDevice, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        rc = cuda_check(ctx, e, "gmres update");
        if (rc) return rc;
        k_update_solution<<<ctx->red_grid, kThreads, 0, s>>>(n, j, ctx->gmV, ctx->gmH, ctx->gmDinv, z);
        ctx->launches++;
        if ((relres <= tol || iters >= max_iter) && !final_check) break;
        if (relres <= tol || iters >= max_iter) {
            // true residual of the final iterate (one more apply)
            rc = bordered_apply(ctx, R, u, sigma, z, w, s, applies > 0);
            if (rc) return rc;
            ++applies;
            relres = residual_norm(ctx, chi, w, w, s, &rc) / bnorm;
            if (rc) return rc;
            break;
        }
    }
    if (info) {
        info->iterations = iters;
        info->applies = applies;
        info->rel_residual = relres;
        double lam = 0.0;
        cudaMemcpyAsync(&lam, z + n, sizeof(double), cudaMemcpyDeviceToHost, s);
        rc = cuda_check(ctx, cudaStreamSynchronize(s), "gmres lambda");
        if (rc) return rc;
        info->lambda = lam;
    }
    return QEQ_OK;
}

namespace {

// Velocity-Verlet half kick and drift; dt / (2 m mass_unit) kept for the second kick.
__global__ void k_kick_drift(int n, double dt, double mass_unit, const double *__restrict__ mass,
                             const double *__restrict__ F, double *__restrict__ R,
                             double *__restrict__ V, double *__restrict__ half_kick) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double hk = 0.5 * dt / (mass[i] * mass_unit);
        half_kick[i] = hk;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const double vi = fma(F[3 * (size_t)i + d], hk, V[3 * (size_t)i + d]);
            V[3 * (size_t)i + d] = vi;
            R[3 * (size_t)i + d] += dt * vi;
        }
    }
}

}  // namespace

int bomd_advance(qeq_ctx *ctx, const qeq_md_params *prm, qeq_md_state *st, cudaStream_t s) {
    const int n = (int)ctx->n;
    prof_begin(ctx, kPhIntegrate, s);
    k_kick_drift<<<ctx->red_grid, kThreads, 0, s>>>(n, ctx->p.dt, ctx->p.mass_unit, prm->mass, st->F,
                                                 st->R, st->V, ctx->half_kick);
    prof_end(ctx, s);
    ctx->launches++;
    double d2 = 0.0;
    int rc = nl_displacement(ctx, st->R, s, &d2);
    if (rc) return rc;
    const double half = 0.5 * ctx->p.skin;
    if (!(d2 <= half * half)) return nl_build(ctx, st->R, s);
    return QEQ_OK;
}

// One BO evaluation at the current positions: solve (warm start from st->q),
// forces F = q o E (+ short range) and energies.  st->q holds N entries; the
// solver's N + 1 vector lives in ctx->gmSol.
int bomd_evaluate(qeq_ctx *ctx, const qeq_md_params *prm, qeq_md_state *st, double tol,
                  int max_iter, qeq_solve_info *info, cudaStream_t s) {
    const int n = (int)ctx->n;
    int rc = solver_alloc(ctx, 40);
    if (rc) return rc;
    if (!ctx->gmSol) {
        rc = dev_alloc(ctx, (void **)&ctx->gmSol, sizeof(double) * (n + 1));
        if (rc) return rc;
        cudaMemsetAsync(ctx->gmSol, 0, sizeof(double) * (n + 1), s);
    }
    cudaMemcpyAsync(ctx->gmSol, st->q, sizeof(double) * n, cudaMemcpyDeviceToDevice, s);
    qeq_solve_info local{};
    // the force apply below evaluates the final charges, so GMRES skips its own check
    rc = gmres_solve(ctx, st->R, prm->chi, prm->eta, prm->sigma, ctx->gmSol, tol, max_iter, 40,
                     false, &local, s);
    if (rc) return rc;
    cudaMemcpyAsync(st->q, ctx->gmSol, sizeof(double) * n, cudaMemcpyDeviceToDevice, s);
    double *scal = ctx->scal;
    rc = short_range_eval(ctx, st->R, prm->mass, scal + 126, s);
    if (rc) return rc;
    // the solve applied the operator at these positions already
    rc = coulomb_apply_impl(ctx, st->R, st->q, prm->sigma, ctx->v_n, ctx->E_n, nullptr, nullptr,
                            true, s, true);
    if (rc) return rc;
    local.applies += 1;
    k_bo_forces<<<ctx->red_grid, kThreads, 0, s>>>(
        n, st->q, ctx->E_n, has_short(ctx) ? ctx->F_short : nullptr, st->F);
    k_bo_energy_part<<<ctx->red_grid, kThreads, 0, s>>>(n, st->q, prm->chi, prm->eta, ctx->v_n, ctx->part);
    launch_finalize(ctx, ctx->part, 4, scal + 128, s);
    k_bo_energies<<<1, 1, 0, s>>>(scal + 128, scal + 126, local.lambda, local.rel_residual,
                                  (double)local.applies, st->energies);
    ctx->launches += 5;
    if (info) *info = local;
    return cuda_check(ctx, cudaGetLastError(), "bomd evaluate launch");
}

}  // namespace qeq
