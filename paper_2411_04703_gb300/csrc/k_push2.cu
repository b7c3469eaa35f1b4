// The dispatcher over the particle kernels' variants (shape order, frozen or mobile, gather scheme,
// region shape), each compiled in a translation unit of its own (k_push1*.cu, k_push2_*.cu), and the charge-density deposit used by pic_get_fields(RHO).
#include "push_impl.cuh"

namespace gbpic {

cudaError_t launch_push1_frozen(pic_ctx *c, int si);
cudaError_t launch_push1_fixed(pic_ctx *c, int si, const ExtDev &ext);
cudaError_t launch_push1_fixed_ec(pic_ctx *c, int si, const ExtDev &ext);
cudaError_t launch_push1_dyn(pic_ctx *c, int si, const ExtDev &ext);
cudaError_t launch_push1_dyn_ec(pic_ctx *c, int si, const ExtDev &ext);
cudaError_t launch_push2_frozen(pic_ctx *c, int si);
cudaError_t launch_push2_fixed(pic_ctx *c, int si, const ExtDev &ext);
cudaError_t launch_push2_fixed_ec(pic_ctx *c, int si, const ExtDev &ext);
cudaError_t launch_push2_dyn(pic_ctx *c, int si, const ExtDev &ext);
cudaError_t launch_push2_dyn_ec(pic_ctx *c, int si, const ExtDev &ext);

namespace {

// Charge density at the nodes: rho += q w S(node - x) / V for every live particle.
template <int ORDER>
__global__ void k_rho(SpeciesDev sp, GridDev g, float qv, float *rho)
{
    using S = push::Shape<ORDER>;
    const int n = sp.count[0];
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        const float4 P = sp.pos[p];
        const int cell = __float_as_int(P.w);
        if (cell < 0) continue;
        const float w = sp.mom[p].w * qv;
        int c[3] = {g.cc.i(cell), g.cc.j(cell), g.cc.k(cell)};
        const int zb = zblock(c[2], g.nzr);
        float o[3] = {P.x, P.y, P.z};
        int su[3];
        float wu[3][S::N];
#pragma unroll
        for (int d = 0; d < 3; d++) S::unst(o[d], su[d], wu[d]);
        for (int k = 0; k < S::N; k++)
            for (int j = 0; j < S::N; j++)
                for (int i = 0; i < S::N; i++) {
                    int q[3] = {c[0] + su[0] + i, c[1] + su[1] + j, c[2] + su[2] + k};
                    bool ok = true;
                    for (int d = 0; d < 2; d++) {
                        if (q[d] < 0 || q[d] >= g.n[d]) {
                            if (g.periodic[d]) q[d] = pwrap(q[d], g.n[d]);
                            else ok = false;
                        }
                    }
                    if (q[2] < zb || q[2] >= zb + g.nzr) {
                        if (g.periodic[2]) q[2] = zb + pwrap(q[2] - zb, g.nzr);
                        else ok = false;
                    }
                    if (ok)
                        atomicAdd(rho + ((long long)q[2] * g.n[1] + q[1]) * g.n[0] + q[0],
                                  w * wu[0][i] * wu[1][j] * wu[2][k]);
                }
    }
}

// Largest displacement per component the stored momenta give in one step, |u_c| dt / (gamma d_c).
__global__ void k_dmax_measure(SpeciesDev sp, float tx, float ty, float tz)
{
    unsigned m[3] = {0u, 0u, 0u};
    const int n = sp.count[0];
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
        if (__float_as_int(sp.pos[p].w) < 0) continue;
        const float4 u = sp.mom[p];
        const float ig = rsqrtf(1.f + u.x * u.x + u.y * u.y + u.z * u.z);
        m[0] = max(m[0], __float_as_uint(fabsf(u.x) * ig * tx));
        m[1] = max(m[1], __float_as_uint(fabsf(u.y) * ig * ty));
        m[2] = max(m[2], __float_as_uint(fabsf(u.z) * ig * tz));
    }
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const unsigned r = __reduce_max_sync(0xffffffffu, m[k]);
        if ((threadIdx.x & 31) == 0 && r) atomicMax(sp.dmax + k, r);
    }
}

// The end of a step in one launch (a dependent launch costs a small grid 2-3 us): the displacement
// bounds of the species pushed, the clock, and the particle kernels' work counters back to zero for the
// next step.
struct StepEnd {
    long long *clock;
    int *work;
    float *dlim[kMaxSpecies];
    unsigned *dmax[kMaxSpecies];
    float light[3];
    int n;
};
__global__ void k_step_end(StepEnd e)
{
    const int q = threadIdx.x, s = q / 3, k = q % 3;
    if (s < e.n) push::dlim_update(e.dlim[s], e.dmax[s], k, k == 0 ? e.light[0] : (k == 1 ? e.light[1] : e.light[2]));
    if (q < 2 * kMaxSpecies && e.work) e.work[q] = 0;
    if (q == 0 && e.clock) *e.clock += 1;
}

void add_dlim(StepEnd &e, const pic_ctx *c, const Species &s)
{
    for (int d = 0; d < 3; d++) e.light[d] = (float)std::min(1.0, c->dt / c->d[d]);
    e.dlim[e.n] = s.dlim;
    e.dmax[e.n++] = s.dmax;
}

}  // namespace

cudaError_t launch_step_end(pic_ctx *c)
{
    static_assert(3 * kMaxSpecies <= 32, "a thread per component of a species");
    StepEnd e{};
    e.clock = c->dclock;
    e.work = c->work;
    for (int si = 0; si < c->nsp; si++)
        if (!c->sp[si].lattice) add_dlim(e, c, c->sp[si]);
    k_step_end<<<1, 32, 0, c->stream>>>(e);
    c->kernels++;
    return cudaGetLastError();
}

// Sets the displacement bound of species si from its current momenta (after a load or an
// injection): four times the largest displacement they give, as after a step.
cudaError_t launch_dlim_from_momenta(pic_ctx *c, int si)
{
    const Species &s = c->sp[si];
    if (s.lattice || !s.dlim) return cudaSuccess;
    k_dmax_measure<<<c->num_sms * 4, 256, 0, c->stream>>>(species_dev(c, s), (float)(c->dt / c->d[0]),
                                                          (float)(c->dt / c->d[1]), (float)(c->dt / c->d[2]));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    StepEnd u{};
    add_dlim(u, c, s);
    k_step_end<<<1, 32, 0, c->stream>>>(u);
    c->kernels += 2;
    return cudaGetLastError();
}

cudaError_t launch_push(pic_ctx *c, int si, const ExtDev &ext)
{
    const bool o1 = c->order == 1;
    if (c->sp[si].frozen) return o1 ? launch_push1_frozen(c, si) : launch_push2_frozen(c, si);
    const bool ec = c->gather == PIC_GATHER_ENERGY;
    if (push::default_region(c)) {
        if (o1) return ec ? launch_push1_fixed_ec(c, si, ext) : launch_push1_fixed(c, si, ext);
        return ec ? launch_push2_fixed_ec(c, si, ext) : launch_push2_fixed(c, si, ext);
    }
    if (o1) return ec ? launch_push1_dyn_ec(c, si, ext) : launch_push1_dyn(c, si, ext);
    return ec ? launch_push2_dyn_ec(c, si, ext) : launch_push2_dyn(c, si, ext);
}

// Adds the charge density of species s to rho.
cudaError_t launch_rho(pic_ctx *c, const Species &s, float *rho)
{
    const float V = (float)(c->d[0] * c->d[1] * c->d[2]);
    const float qv = (float)(s.q / V);
    if (c->order == 1) k_rho<1><<<c->num_sms * 8, 256, 0, c->stream>>>(species_dev(c, s), grid_dev(c), qv, rho);
    else k_rho<2><<<c->num_sms * 8, 256, 0, c->stream>>>(species_dev(c, s), grid_dev(c), qv, rho);
    c->kernels++;
    return cudaGetLastError();
}

}  // namespace gbpic
