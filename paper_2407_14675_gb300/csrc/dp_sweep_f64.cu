// Sweep kernels with double geometry and double values.
#include "dp_sweep.cuh"

namespace dpk {

cudaError_t launch_sweep(const SweepLaunch<double, double>& L)
{
    if (L.dyn == kDynUnitSpeed) {
        if (L.reduced) return cudaErrorInvalidValue;
        return launch_mode<double, double, kDynUnitSpeed, false>(L);
    }
    if (L.dyn == kDynPolar) {
        if (L.reduced) return cudaErrorInvalidValue;
        return launch_mode<double, double, kDynPolar, false>(L);
    }
    if (L.reduced) return launch_mode<double, double, kDynOrbit, true>(L);
    return launch_mode<double, double, kDynOrbit, false>(L);
}

// The parts of node_dyn() that a row (i_r, i_vr) or a mass node shares, with its
// operations, the node coordinates, and (polar) dt times the running cost.
__global__ void dyn_tables_kernel(const Geo<double> g, double2* rows, double2* mass, double* coord, double* cost)
{
    const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const bool polar = g.dyn == kDynPolar;
    if (t < (long long)g.n[0] * g.n[1]) {
        const int i0 = (int)(t / g.n[1]), i1 = (int)(t % g.n[1]);
        const double r = g.lo[0] + (double)i0 * g.h[0], vr = g.lo[1] + (double)i1 * g.h[1];
        const double ir = grcp(r), ir2 = grcp(xfma(g.dt, vr, r));
        rows[2 * t] = make_double2(ir, xmul(g.mu, xmul(ir, ir)));
        rows[2 * t + 1] = make_double2(ir2, xmul(g.mu, xmul(ir2, ir2)));
    }
    if (t < (polar ? 1 : g.n[3])) {
        double am = g.accel, am2 = g.accel;
        if (!polar) {
            const double m = g.lo[3] + (double)t * g.h[3];
            am = xmul(g.accel, grcp(m));
            am2 = xmul(g.accel, grcp(xfma(g.dt, g.mdot, m)));
        }
        const double R1 = xmul(g.dt, am), amm = xadd(am, am2);
        mass[2 * t] = make_double2(R1, amm);
        mass[2 * t + 1] = make_double2(xmul(g.hh[0], R1), xmul(g.hh[1], amm));
    }
    if (t < 4 * kCoordStride) {
        const int d = (int)(t / kCoordStride), i = (int)(t % kCoordStride);
        if (i < g.n[d]) coord[t] = g.lo[d] + (double)i * g.h[d];
    }
    if (cost && t < g.n_nodes) {
        int i[4];
        decode_node(g, (int)t, i);
        cost[t] = __dmul_rn(g.dt64, state_cost(g, i));
    }
}

cudaError_t launch_dyn_tables(const Geo<double>& g, double2* rows, double2* mass, double* coord, double* cost,
                              cudaStream_t st)
{
    long long n = (long long)g.n[0] * g.n[1];
    if (n < 4 * kCoordStride) n = 4 * kCoordStride;
    if (cost && n < g.n_nodes) n = g.n_nodes;
    dyn_tables_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(g, rows, mass, coord, cost);
    return cudaGetLastError();
}

}  // namespace dpk
