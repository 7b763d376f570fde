// imb_adjoint.cu -- reverse-mode gradient of the time-averaged drag on fixed disks.
//
// The forward step is the stream-collide kernel: f(t) = pull(P(t-1)) with the boundary
// rules (Eq. 1 LHS), P(t) = collision of f(t) (Eqs. 1-2, 12-14), drag D(t) = sum_p F_x,p
// (Eq. 15).  For disks at rest, plain BGK and no body force the solid term summed over a
// cell's disks is B (f_{-i} - f^eq_{-i}(rho, u) + w_i rho - f_i) and the cell's drag is
// B j_x, so J = (1/T) sum_t D(t) depends on the disk positions only through the summed
// solid ratio E of each cell.  Going backwards in time, one kernel per step
//   * gathers the adjoint of P(t) from the adjoint of f(t+1) (the transpose of the pull:
//     a gather at x + c_i, bounce-back entries from the cell itself),
//   * recomputes f(t) from P(t-1) and applies the transposed Jacobian of the collision
//     (plus the drag's own dependence on f),
//   * adds d J / d tau and d J / d E of the cell.
//   * transposes the inlet and outlet columns of the pull (f(0) = f^eq(rho of column 1, u_in),
//     f(nx-1) = f^eq(1, u of column nx-2)), adding d J / d u_in.
// d E / d (disk centre) is the difference of the chord lengths on opposite cell edges.
#include "imb_device.cuh"
#include "imb_host.h"
#include "imb_kernels.h"
#include "imb_sums.h"
#include "imb_pull.cuh"

namespace imb {

// J: the drag that k_step_tail summed over the steps, particle by particle, over the particles
__global__ void __launch_bounds__(256) k_drag_sum(const double *__restrict__ Jsum, int np, double *acc) {
    __shared__ double s[8];
    double v = 0.0;
    for (int p = threadIdx.x; p < np; p += 256) v += Jsum[p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < 8; ++w) t += s[w];
        *acc += t;
    }
}

// summed solid ratio of every cell, in slot order (the order the collision sums them)
__global__ void k_cell_E(const int *__restrict__ count, const float *__restrict__ eps, size_t ncell, float *E) {
    const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= ncell) return;
    float e = 0.0f;
    for (int k = 0; k < count[c]; ++k) e += eps[c * MAX_SLOTS + k];
    E[c] = e;
}

// sum of the nine directions, in the order of a butterfly over lanes
__device__ __forceinline__ float tree9(const float (&v)[9]) {
    return (((v[0] + v[8]) + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
}

// One step backwards: lam1 = d J / d f(t+1) (columns already transposed), S0 = P(t-1)
// (f(t) is pulled from it); writes lam0 = d J / d f(t).  With `inlet` the transpose of the inlet
// and outlet columns of the pull that gave f(t) from S0 follows in the same launch: f(0) =
// f^eq(rho of column 1, u_in) and f(nx-1) = f^eq(1, u of column nx-2) hand the adjoint of columns 0
// and nx - 1 on to the threads of columns 1 and nx - 2, which hold the pulled f(t) they need, and
// the row's d J / d u_in to g_uin (columns 0 and 1, and nx - 2 and nx - 1, share a block: adjoint_grid).
//
// d J / d tau is summed over the block in three FP32 parts (Sum3: an FP64 add takes a warp 64 cycles, and
// every warp's shuffle tree took five of them; even the three conversions at the end of each warp's sum
// kept the FP64 pipe busy for 29 % of the launch on 2048 x 1024 cells, 71 us against 67).  What leaves
// FP32's range is summed in FP64.  The adjoint itself keeps the order of its sums:
// taken on opposite pairs it has fewer instructions and is no faster on 512 x 256 cells (43 us a
// forward and reverse step, 84 before the launches and copies were saved), but where the adjoint front
// has not reached the inlet d J / d u_in is rounding noise, which any other order changes whole.
__global__ void __launch_bounds__(ADJ_BLOCK) k_adjoint_step(const float *__restrict__ lam1, const float *__restrict__ S0,
                                                      float *__restrict__ lam0, const LatticeArgs a,
                                                      const float *__restrict__ E, double *__restrict__ gE,
                                                      float inv_T, double *g_tau, int inlet, double *g_uin, int shift) {
    cudaGridDependencySynchronize();   // launched as a dependent of the kernel before it
    cudaTriggerProgrammaticLaunchCompletion();
    __shared__ float edge[2][9];
    __shared__ float part[3][ADJ_BLOCK / 32];
    __shared__ double part64[ADJ_BLOCK / 32];
    const int x = (int)(blockIdx.x * blockDim.x + threadIdx.x) - shift, y = blockIdx.y;
    const bool in = x >= 0 && x < a.nx;
    float gt = 0.0f, gt_B = 0.0f;   // the cell's d J / d tau, and through B
    lam1 += a.origin;   // node (0, 0) of plane 0 in the frame
    S0 += a.origin;
    lam0 += a.origin;
    float v[9];
    float col_rho = 1.0f, col_ux = 0.0f, col_uy = 0.0f;
    if (in) {
        // adjoint of P(t) at (x, y): who pulled P_q(x, y); and f(t) at (x, y), pulled from
        // P(t-1) (shifted populations d = f - w).  Away from the edges no boundary rule applies.
        float L[9], d[9];
        const size_t c = (size_t)y * a.nx + x;
        const float Ec = E[c];
        const bool inner = x >= 1 && x <= a.nx - 2 && y >= 1 && y <= a.ny - 2;
        if (inner) {
            const size_t c0 = (size_t)y * a.pitch + x;
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const ptrdiff_t off = (ptrdiff_t)cy_of(q) * a.pitch + cx_of(q);
                L[q] = lam1[(size_t)q * a.plane + c0 + off];
                d[q] = S0[(size_t)q * a.plane + c0 - off];
            }
        } else {
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                int xd = x + cx_of(q), yd = y + cy_of(q);
                bool bounce = false, gone = false;
                if (yd < 0 || yd >= a.ny) {
                    if (a.bc_y == BC_PERIODIC) yd = yd < 0 ? yd + a.ny : yd - a.ny;
                    else bounce = true;
                }
                if (!bounce && (xd < 0 || xd >= a.nx)) {
                    if (a.bc_x == BC_PERIODIC) xd = xd < 0 ? xd + a.nx : xd - a.nx;
                    else if (a.bc_x == BC_WALL) bounce = true;
                    else gone = true;
                }
                L[q] = gone ? 0.0f
                       : bounce ? lam1[(size_t)opp_of(q) * a.plane + (size_t)y * a.pitch + x]
                                : lam1[(size_t)q * a.plane + (size_t)yd * a.pitch + xd];
            }
            pull_cell(S0, a, x, y, d);
        }
        float drho = 0.0f, jx = 0.0f, jy = 0.0f;
#pragma unroll
        for (int q = 0; q < 9; ++q) {   // products with a zero velocity component left out
            drho += d[q];
            if (cx_of(q) != 0) jx += cx_of(q) > 0 ? d[q] : -d[q];
            if (cy_of(q) != 0) jy += cy_of(q) > 0 ? d[q] : -d[q];
        }
        const float rho = 1.0f + drho, ux = jx / rho, uy = jy / rho, usq = ux * ux + uy * uy;
        float n[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float cu = cdot(q, ux, uy);
            n[q] = d[q] - w_of(q) * (drho + rho * (3.0f * cu + 4.5f * cu * cu - 1.5f * usq));
        }
        const float e = fminf(Ec, 1.0f), tau = a.tau, tm = tau - 0.5f;
        const float B = Ec > 0.0f ? e * tm / ((1.0f - e) + tm) : 0.0f;
        const float af = (1.0f - B) / tau;
        float mu[9], nu = 0.0f;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            mu[q] = af * L[q] - B * L[opp_of(q)];
            nu += B * w_of(q) * L[q];
        }
        float lr = nu, ljx = 0.0f, ljy = 0.0f;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float cxq = (float)cx_of(q), cyq = (float)cy_of(q), cu = cdot(q, ux, uy);
            lr += mu[q] * w_of(q) * (1.0f - 4.5f * cu * cu + 1.5f * usq);
            ljx += mu[q] * w_of(q) * (cx_of(q) != 0 ? 3.0f * cxq + 9.0f * cu * cxq - 3.0f * ux : -3.0f * ux);
            ljy += mu[q] * w_of(q) * (cy_of(q) != 0 ? 3.0f * cyq + 9.0f * cu * cyq - 3.0f * uy : -3.0f * uy);
        }
        float Ln = 0.0f;
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            const float cxq = (float)cx_of(q), cyq = (float)cy_of(q);
            float t = L[q] * (1.0f - af - B) + B * L[opp_of(q)];
            if (cx_of(q) != 0) t += inv_T * B * cxq;
            t += lr;
            if (cx_of(q) != 0) t += cxq * ljx;
            if (cy_of(q) != 0) t += cyq * ljy;
            v[q] = t;
            Ln += L[q] * (1.0f - B) * n[q];
        }
        gt = Ln / (tau * tau);
        if (B > 0.0f) {
            float lB = inv_T * jx;
#pragma unroll
            for (int q = 0; q < 9; ++q) lB += L[q] * (n[q] / tau + n[opp_of(q)] + w_of(q) * drho - d[q]);
            const float den = (1.0f - e) + tm;
            gt_B = lB * e * (1.0f - e) / (den * den);
            if (Ec < 1.0f) gE[c] += (double)(lB * tm * (1.0f + tm) / (den * den));
        }
        if (inlet && (x == 1 || x == a.nx - 2)) {   // f(t) of the column, for the columns next to it
            float mx[9], my[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                mx[q] = (float)cx_of(q) * d[q];
                my[q] = (float)cy_of(q) * d[q];
            }
            col_rho = 1.0f + tree9(d);
            col_ux = tree9(mx) / col_rho;
            col_uy = tree9(my) / col_rho;
        }
    }
    if (inlet && (blockIdx.x == 0 || blockIdx.x == gridDim.x - 1)) {
        if (x == 0 || x == a.nx - 1)
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                edge[x == 0 ? 0 : 1][q] = v[q];
                v[q] = 0.0f;
            }
        __syncthreads();
        if (x == a.nx - 2) {
            // outlet: f(nx-1) = f^eq(1, u), u = j / rho of f(nx-2); d f^eq_q / d u = w_q (3 c_q +
            // 9 (c_q . u) c_q - 3 u), d u / d f_p(nx-2) = (c_p - u) / rho
            const float rho = col_rho, ux = col_ux, uy = col_uy;
            float px[9], py[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const float cxq = (float)cx_of(q), cyq = (float)cy_of(q), lo = edge[1][q], wq = w_of(q);
                const float cu = cxq * ux + cyq * uy;
                px[q] = lo * wq * (3.0f * cxq + __fmul_rn(9.0f, cu) * cxq - 3.0f * ux);
                py[q] = lo * wq * (3.0f * cyq + __fmul_rn(9.0f, cu) * cyq - 3.0f * uy);
            }
            const float gx = tree9(px), gy = tree9(py);
#pragma unroll
            for (int q = 0; q < 9; ++q) v[q] += (gx * ((float)cx_of(q) - ux) + gy * ((float)cy_of(q) - uy)) / rho;
        }
        if (x == 1) {   // inlet: f(0) = f^eq(rho1, u_in), rho1 = 1 + the pulled shifted populations of column 1
            const float ux = a.u_in_x, uy = a.u_in_y, usq = ux * ux + uy * uy;
            float pr[9], pg[9];
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const float cxq = (float)cx_of(q), cyq = (float)cy_of(q), l0 = edge[0][q], wq = w_of(q);
                const float cu = cxq * ux + cyq * uy;
                pr[q] = l0 * wq * (1.0f + 3.0f * cu + 4.5f * cu * cu - 1.5f * usq);
                pg[q] = l0 * wq * (3.0f * cxq + __fmul_rn(9.0f, cu) * cxq - 3.0f * ux);
            }
            const float l = tree9(pr), g = tree9(pg);
#pragma unroll
            for (int q = 0; q < 9; ++q) v[q] += l;
            if (g != 0.0f) atomicAdd(g_uin, (double)(g * col_rho));
        }
    }
    if (in) {
#pragma unroll
        for (int q = 0; q < 9; ++q) lam0[(size_t)q * a.plane + (size_t)y * a.pitch + x] = v[q];
    }
    Sum3 sum;
    sum.add(gt);
    sum.add(gt_B);
    auto join = [&](int from) {
#pragma unroll
        for (int o = from; o > 0; o >>= 1) {
            Sum3 other;
            other.hi = __shfl_xor_sync(0xffffffffu, sum.hi, o);
            other.lo = __shfl_xor_sync(0xffffffffu, sum.lo, o);
            other.lo2 = __shfl_xor_sync(0xffffffffu, sum.lo2, o);
            sum.add(other);
        }
    };
    join(16);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (__any_sync(0xffffffffu, !sum.finite())) {   // a sum beyond FP32, an infinity or NaN
        double t = (double)gt + (double)gt_B;
        for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) part64[warp] = t;
    }
    if (lane == 0) {
        part[0][warp] = sum.hi;
        part[1][warp] = sum.lo;
        part[2][warp] = sum.lo2;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        constexpr int WARPS = ADJ_BLOCK / 32;
        auto of_warp = [&](int w) {
            Sum3 p;
            if (w < WARPS) {
                p.hi = part[0][w];
                p.lo = part[1][w];
                p.lo2 = part[2][w];
            }
            return p;
        };
        sum = of_warp(lane);
        join(WARPS / 2);
        if (lane == 0 && !(sum.hi == 0.0f && sum.lo == 0.0f)) {
            double t = sum.value();
            if (!sum.finite()) {
                t = 0.0;
                for (int w = 0; w < WARPS; ++w) t += of_warp(w).finite() ? of_warp(w).value() : part64[w];
            }
            atomicAdd(g_tau, t);
        }
    }
}

// vertical chord of a disk centred at the origin on the line x = a, within [b0, b1]
__device__ __forceinline__ double chord_len(double a, double b0, double b1, double r) {
    if (!(fabs(a) < r)) return 0.0;
    const double h = sqrt(r * r - a * a);
    const double lo = fmax(b0, -h), hi = fmin(b1, h);
    return hi > lo ? hi - lo : 0.0;
}

// d J / d (disk centre) = sum over the cells a disk covers of d J / d E times d E / d centre
__global__ void k_position_grad(const int *__restrict__ count, const int *__restrict__ ids,
                                const double *__restrict__ gE, const double *__restrict__ xp,
                                const double *__restrict__ rp, int nx, int ny, int bc_x, int bc_y,
                                double *dJ_dx) {
    const size_t c = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= (size_t)nx * ny || count[c] == 0 || gE[c] == 0.0) return;
    const int i = (int)(c % nx), k = (int)(c / nx);
    for (int sl = 0; sl < count[c]; ++sl) {
        const int p = ids[c * MAX_SLOTS + sl];
        const double cx = xp[2 * p], cy = xp[2 * p + 1], r = rp[p];
        double ax = (double)i - cx, ay = (double)k - cy;   // cell corner relative to the centre
        if (bc_x == BC_PERIODIC) ax -= nx * rint(ax / nx);
        if (bc_y == BC_PERIODIC) ay -= ny * rint(ay / ny);
        // moving the centre by +d moves the cell by -d relative to the disk
        const double gx = chord_len(ax, ay, ay + 1.0, r) - chord_len(ax + 1.0, ay, ay + 1.0, r);
        const double gy = chord_len(ay, ax, ax + 1.0, r) - chord_len(ay + 1.0, ax, ax + 1.0, r);
        atomicAdd(&dJ_dx[2 * p], gE[c] * gx);
        atomicAdd(&dJ_dx[2 * p + 1], gE[c] * gy);
    }
}

cudaError_t launch_drag_sum(const double *Jsum, int np, double *acc, cudaStream_t s) {
    k_drag_sum<<<1, 256, 0, s>>>(Jsum, np, acc);
    return cudaGetLastError();
}

cudaError_t launch_cell_E(const int *count, const float *eps, size_t ncell, float *E, cudaStream_t s) {
    k_cell_E<<<(unsigned)((ncell + 255) / 256), 256, 0, s>>>(count, eps, ncell, E);
    return cudaGetLastError();
}

cudaError_t launch_adjoint_step(const float *lam1, const float *S0, float *lam0, const LatticeArgs &a,
                                const float *E, double *gE, float inv_T, double *g_tau, bool inlet, double *g_uin,
                                cudaStream_t s) {
    const AdjointGrid g = adjoint_grid(a.nx, inlet);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(g.blocks, a.ny);
    cfg.blockDim = dim3(ADJ_BLOCK);
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_adjoint_step, lam1, S0, lam0, a, E, gE, inv_T, g_tau, (int)inlet, g_uin, g.shift);
}

cudaError_t launch_position_grad(const int *count, const int *ids, const double *gE, const double *x,
                                 const double *r, int nx, int ny, int bc_x, int bc_y, double *dJ_dx,
                                 cudaStream_t s) {
    const size_t n = (size_t)nx * ny;
    k_position_grad<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(count, ids, gE, x, r, nx, ny, bc_x, bc_y, dJ_dx);
    return cudaGetLastError();
}

}  // namespace imb
