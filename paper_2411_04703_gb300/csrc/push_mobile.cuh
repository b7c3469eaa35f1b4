// Particle kernel of the mobile species (sm_103a): gather, external field, push, move and Esirkepov
// deposit.
#pragma once

#include "push_impl.cuh"

namespace gbpic {
namespace push {

__device__ __forceinline__ void cp_async4(void *dst, const void *src)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16(void *dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// Shape values and differences on the simple window by the general window's formulas: what
// deposit_general forms at these nodes, bit by bit (beyond them it holds zeros while the nearest node
// stays).  A cold lattice crosses all at once and rounds alike, and its electrons' and ions' currents
// nearly cancel: a crossing particle's current keeps the form it has on every other path (2 % of the
// kernel where a quarter of the particles cross).
template <int ORDER>
__device__ __forceinline__ void shapes_general(float o, float d, int &st, float S0[ORDER + 1], float DS[ORDER + 1])
{
    using S = Shape<ORDER>;
    st = ORDER == 2 ? (o >= 0.5f ? 0 : -1) : 0;
#pragma unroll
    for (int a = 0; a <= ORDER; a++) {
        S0[a] = S::S(o - (float)(st + a));
        DS[a] = S::seg(o, st + a, d, d, 1.f);
    }
}

// Deposit of a particle whose nearest node (TSC) or cell (CIC) changes along one dim only (e): the
// window is a node longer along e than the simple one and as long along the two others, 75 nodes for
// TSC against the general window's 144 and without the general window's tests at every node.  The
// dims are taken in the cyclic order e, e + 1, e + 2 with their strides, so one code serves all.  The
// prefix over the simple window's last node is the rounding of its sum, which the general window
// deposits too where it isn't zero.
template <int ORDER, class Reg>
__device__ __forceinline__ void deposit_cross(const SmemAcc<Reg> &acc, const float o[3], const float d[3], const int s[3],
                                              const float fac[3], int e, const float v[3], const float h[3])
{
    using S = Shape<ORDER>;
    constexpr int L = S::L, N = S::N;
    const int stride[3] = {1, acc.reg.rx(), acc.reg.r2()};
    const int a = e == 2 ? 0 : e + 1, b = a == 2 ? 0 : a + 1;
    auto pickf = [](const auto *p, int i) { return i == 0 ? p[0] : (i == 1 ? p[1] : p[2]); };
    const int se = pickf(stride, e), sa = pickf(stride, a), sb = pickf(stride, b);
    const float oe = pickf(o, e), de = pickf(d, e);
    const int she = pickf(s, e);
    float S0e[L], De[L], S0a[N], Da[N], S0b[N], Db[N];
    int ste, sta, stb;
    S::general(oe, de, she, pickf(v, e), pickf(h, e), ste, S0e, De);
    shapes_general<ORDER>(pickf(o, a), pickf(d, a), sta, S0a, Da);
    shapes_general<ORDER>(pickf(o, b), pickf(d, b), stb, S0b, Db);
    float Ae[L], Qe[L], Fe[L - 1], Aa[N], Qa[N], Fa[N], Ab[N], Qb[N], Fb[N];
    const float fe = pickf(fac, e) * acc.scale(e), fa = pickf(fac, a) * acc.scale(a), fb = pickf(fac, b) * acc.scale(b);
    float run = 0.f;
#pragma unroll
    for (int i = 0; i < L; i++) {
        Ae[i] = fmaf(0.5f, De[i], S0e[i]);
        Qe[i] = De[i] * (1.f / 12.f);
        run += De[i];
        if (i < L - 1) Fe[i] = fe * run;
    }
    float ra = 0.f, rb = 0.f;
#pragma unroll
    for (int i = 0; i < N; i++) {
        Aa[i] = fmaf(0.5f, Da[i], S0a[i]);
        Qa[i] = Da[i] * (1.f / 12.f);
        Ab[i] = fmaf(0.5f, Db[i], S0b[i]);
        Qb[i] = Db[i] * (1.f / 12.f);
        ra += Da[i];
        rb += Db[i];
        Fa[i] = fa * ra;
        Fb[i] = fb * rb;
    }
    const int at = acc.base + ste * se + sta * sa + stb * sb;
    const int pe = at + e * acc.reg.r3(), pa = at + a * acc.reg.r3(), pb = at + b * acc.reg.r3();
#pragma unroll
    for (int m = 0; m < N; m++)
#pragma unroll
        for (int l = 0; l < N; l++) {
            const float Y = fmaf(Aa[l], Ab[m], Qa[l] * Db[m]);
#pragma unroll
            for (int k = 0; k < L - 1; k++) acc.add(pe + k * se + l * sa + m * sb, Fe[k] * Y);
        }
#pragma unroll
    for (int m = 0; m < L; m++)
#pragma unroll
        for (int l = 0; l < N; l++) {
            const float Ya = fmaf(Ab[l], Ae[m], Qb[l] * De[m]);       // J_a: a; b, e
            const float Yb = fmaf(Ae[m], Aa[l], Qe[m] * Da[l]);       // J_b: b; e, a
#pragma unroll
            for (int k = 0; k < N - 1; k++) {
                acc.add(pa + k * sa + l * sb + m * se, Fa[k] * Ya);
                acc.add(pb + k * sb + l * sa + m * se, Fb[k] * Yb);
            }
            if (Fa[N - 1] != 0.f) acc.add(pa + (N - 1) * sa + l * sb + m * se, Fa[N - 1] * Ya);
            if (Fb[N - 1] != 0.f) acc.add(pb + (N - 1) * sb + l * sa + m * se, Fb[N - 1] * Yb);
        }
}

// ------------------------------------------------------------------ the kernel
// A work item is up to kChunk particles of one tile.  Its E and B region is staged in shared memory
// and its current summed there in fixed point (see SmemAcc), as for the frozen species; a thread
// takes one particle at a time.  The bound is the shared-memory and L1 pipe together with issue: per
// particle 162 field loads, 108 atomics and the records' lines against ~1,500 thread instructions.
//  - Lanes: the sort leaves a tile's particles octant by octant along its rows (tile_key), so that
//    32 consecutive records of a lattice are on 32 cells at the same place in their cells.  Lane l
//    takes record l K + k, K the records of an octant in an even tile: for K = 1 a warp's records
//    fill whole lines and its 8 x 4 cells 32 different banks (push_pitch); a denser tile spreads its
//    lanes over more cells instead of queueing them on the same words.  With the records of a cell
//    together (lanes 128 records apart) every record was a line of its own, one line a clock, and
//    field loads and atomics met 1.5 and 1.7 times: 20 clocks a particle on that pipe, now 13.
//  - The region spans the nodes that gathers and simple deposits touch, a node less on each side
//    than the general deposit window needs (13^3 instead of 15^3 for TSC on 8^3 cells).
//  - The region starts at the tile's edge less the margin unless the particles can have drifted
//    further than that since the sort: it then follows the item's particles, as long as they fit.
//  - Particles whose nearest node changes in the step are listed and taken after the others, a thread
//    each: nearly all change it along one dim (deposit_cross).  So are particles outside the region,
//    through global memory.
//  - Two CTAs of the default tile's region fit on an SM, so that one stages, flushes or waits while
//    the other computes (the list shares the fields' memory, the marks are a bit a record).  The next
//    item's number and record are fetched behind the present one's staging, and a flush leaves the
//    currents' words zero (300k electrons 0.113 -> 0.110 ms per step).
// ms per step, with the cell-ordered lanes -> now: plasma buncher 5.22 -> 4.24, sweep of 64 runs 18.0 ->
// 15.9, long undulator 4.66 -> 4.18, 65k electrons CIC 0.045 -> 0.028 (the region follows the drift), 2-D
// buncher 2.40 -> 1.75.  (Two CTAs for the plasmas: 3.80, 13.6, and 1.18 with four in 2-D; see INORDER.)
//
// NEUTRAL: a species whose current another one's nearly cancels (see cancels).
//  - Its crossings' last digit shows in the fields (see Shape), and a lattice that crosses takes its tiles'
//    currents with it.  An item's first kQueue crossings are formed from the rounded displacement, the
//    rest from the product it rounds, in the order of gq passes over the octants: 1.2e-3 of E lies between
//    that and one form for all, for a lattice of 2 x 2 x 2 a cell of which half crosses.
// INORDER: its tiles' currents are added to the other's, each addition rounded at that one's size, so a
// shared node depends on which of its tiles flushes first.  With one CTA an SM, and an item claimed when
// the one before it is flushed, neighbours flush in the order of the items.  An item claimed ahead lets
// the CTAs drift apart, and two CTAs flush twice as many tiles at once: two launches of one state then
// differ 2 to 4 times as much (J of 76 x 78 x 298 cells at 4 a cell, 4 steps: 1.4e-5, 6.4e-5 so).
template <int ORDER, int GATHER, int NT, int MINB, bool NEUTRAL, bool INORDER, class Reg>
__global__ void __launch_bounds__(NT, MINB)
k_push(SpeciesDev sp, GridDev g, TileDev t, FieldsDev f, ExtDev ext0, int *work, int *work_sparse, int *err, Reg reg, int age)
{
    using S = Shape<ORDER>;
    const ExtDev ext = ext_at_clock(ext0);
    extern __shared__ __align__(16) float smem[];
    __shared__ int4 s_item;
    __shared__ float s_js[3], s_jinv[3], s_dl[3];
    __shared__ int s_lo[3], s_hi[3], s_sum[3], s_live, s_n;
    constexpr int PASSES = NEUTRAL ? 2 : 1;
    __shared__ unsigned s_mark[PASSES][kChunk / 32];   // listed records, a bit each (in the order of the passes)
    const int Rx = reg.rx(), Ry = reg.ry(), R2 = reg.r2(), R3 = reg.r3(), Rz = R3 / R2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // dynamic shared memory: the currents' words and the fields; the list takes the fields' place when
    // every particle is pushed (two CTAs of the 13^3 region then fit on an SM, to 300 bytes)
    unsigned *sJlo = reinterpret_cast<unsigned *>(smem);
    int *sJhi = reinterpret_cast<int *>(sJlo + 3 * R3);
    float *sF = reinterpret_cast<float *>(sJhi + 3 * R3);
    unsigned short *list = reinterpret_cast<unsigned short *>(sF);

    const int n_total = sp.count[0], n_sorted = sp.count[1], n_items = sp.count[2];
    const long long gnx = g.n[0], gnxy = (long long)g.n[0] * g.n[1];
    unsigned dmax[3] = {0u, 0u, 0u};

    auto claim = [&]() {
        const int it = atomicAdd(work, 1);
        s_item = it < n_items ? t.items[it] : make_int4(-1, 0, 0, 0);
    };
    if (!INORDER && tid == 0) claim();
    for (int l = tid; l < 6 * R3; l += NT) sJlo[l] = 0u;   // both words; a flush leaves them zero again
    for (;;) {
        if (tid == 0) {
            if (INORDER) claim();
            else cp_async_wait();                  // s_item
            s_n = 0;
            s_live = 0;
        }
        for (int l = tid; l < PASSES * (kChunk / 32); l += NT) s_mark[0][l] = 0u;
        if (tid < 3) {
            s_lo[tid] = 1 << 20;
            s_hi[tid] = -(1 << 20);
            s_sum[tid] = 0;
        }
        __syncthreads();
        const int4 item = s_item;
        if (item.x < 0) break;
        int it = 0;
        if (!INORDER && tid == 0) it = atomicAdd(work, 1);   // the next item's number, and behind the staging its record
        const int tile = item.x, p0 = item.y, p1 = item.z;
        const int t0[3] = {(tile % t.nt[0]) * t.T[0], ((tile / t.nt[0]) % t.nt[1]) * t.T[1], (tile / (t.nt[0] * t.nt[1])) * t.T[2]};
        const int zb = g.nzr == g.n[2] ? 0 : zblock(t0[2], g.nzr);
        // cell coordinates relative to the tile (the nearest periodic image)
        auto relative = [&](int cell, int rel[3]) {
            const int c[3] = {g.cc.i(cell), g.cc.j(cell), g.cc.k(cell)};
#pragma unroll
            for (int d = 0; d < 3; d++) {
                int r = c[d] - t0[d];
                if (g.periodic[d]) {
                    const int per = d == 2 ? g.nzr : g.n[d];
                    if (r > per / 2) r -= per;
                    else if (r < -per / 2) r += per;
                }
                rel[d] = r;
            }
        };
        if (tid < 3) {
            // fixed-point scale of the item: the largest contribution jb w dlim maps to <= 2^30
            const float w = sp.wrun ? sp.wrun[t0[2] / g.nzr] : sp.wmax;
            const float dl = sp.dlim[tid];
            const float bd = sp.jb[tid] * w * dl;
            int e = 0;
            frexpf(bd, &e);                       // bd < 2^e
            const int ex = bd > 0.f ? min(max(30 - e, -100), 100) : 0;
            s_js[tid] = ldexpf(1.f, ex);
            s_jinv[tid] = ldexpf(1.f, -ex);
            s_dl[tid] = dl;
        }
        int org[3] = {-t.M, -t.M, -t.M};
        // (dlim bounds a step's displacement: four times the last step's largest, at most light's)
        const float reach = (float)age * fmaxf(sp.dlim[0], fmaxf(sp.dlim[1], sp.dlim[2]));
        if (reach > (float)t.M) {
            int lo[3] = {1 << 20, 1 << 20, 1 << 20}, hi[3] = {-(1 << 20), -(1 << 20), -(1 << 20)}, sum[3] = {0, 0, 0}, live = 0;
            for (int p = p0 + tid; p < p1; p += NT) {
                const int cell = __float_as_int(sp.pos[p].w);
                if (cell < 0) continue;
                int rel[3];
                relative(cell, rel);
#pragma unroll
                for (int d = 0; d < 3; d++) {
                    lo[d] = min(lo[d], rel[d]);
                    hi[d] = max(hi[d], rel[d]);
                    sum[d] += rel[d];
                }
                live++;
            }
            live = __reduce_add_sync(0xffffffffu, live);
            if (lane == 0) atomicAdd(&s_live, live);
#pragma unroll
            for (int d = 0; d < 3; d++) {
                lo[d] = __reduce_min_sync(0xffffffffu, lo[d]);
                hi[d] = __reduce_max_sync(0xffffffffu, hi[d]);
                sum[d] = __reduce_add_sync(0xffffffffu, sum[d]);
                if (lane == 0) {
                    atomicMin(&s_lo[d], lo[d]);
                    atomicMax(&s_hi[d], hi[d]);
                    atomicAdd(&s_sum[d], sum[d]);
                }
            }
            __syncthreads();
#pragma unroll
            for (int d = 0; d < 3; d++) {
                const int w = t.T[d] + 2 * t.M, l = s_lo[d], h = s_hi[d];
                if (h < l) continue;
                if (h - l + 1 > w) org[d] = (int)floorf((float)s_sum[d] / (float)s_live + 1.f) - w / 2;   // about their mean
                else if (l < org[d]) org[d] = l;
                else if (h >= org[d] + w) org[d] = h - w + 1;
            }
        }
        const int reg0[3] = {t0[0] + org[0] - 1, t0[1] + org[1] - 1, t0[2] + org[2] - 1};
        const bool interior = reg0[0] >= 0 && reg0[0] + Rx <= g.n[0] && reg0[1] >= 0 && reg0[1] + Ry <= g.n[1] &&
                              reg0[2] >= zb && reg0[2] + Rz <= zb + g.nzr;
        const long long gbase = reg0[2] * gnxy + reg0[1] * gnx + reg0[0];
        auto node = [&](int l) {
            const int lz = l / R2, rem = l - lz * R2, ly = rem / Rx, lx = rem - ly * Rx;
            if (ly >= Ry) return -1ll;               // plane padding
            return interior ? gbase + lz * gnxy + ly * gnx + lx : wrap_node(g, reg0[0] + lx, reg0[1] + ly, reg0[2] + lz, zb);
        };
        for (int l = tid; l < R3; l += NT) {
            const long long gi = node(l);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                if (gi >= 0) {
                    cp_async4(sF + c * R3 + l, f.E + c * g.ncell + gi);
                    cp_async4(sF + (c + 3) * R3 + l, f.B + c * g.ncell + gi);
                } else {
                    sF[c * R3 + l] = 0.f;
                    sF[(c + 3) * R3 + l] = 0.f;
                }
            }
        }
        cp_async_wait();
        __syncthreads();
        if (!INORDER && tid == 0) {
            if (it < n_items) cp_async16(&s_item, t.items + it);
            else s_item.x = -1;
        }

        // region coordinates of a cell: true inside the region
        auto in_region = [&](int cell, int rel[3]) {
            relative(cell, rel);
            bool in = true;
#pragma unroll
            for (int d = 0; d < 3; d++) {
                rel[d] -= org[d];
                in = in && (unsigned)rel[d] < (unsigned)(t.T[d] + 2 * t.M);
                rel[d] += 1;
            }
            return in;
        };
        const int len = p1 - p0;
        const int gq = (len + kQueue - 1) / kQueue;
        const int K = max(1, min((item.w + 4 * t.tile_cells) / (8 * t.tile_cells), (len + 31) / 32));
        const int rounds = (len + 32 * K - 1) / (32 * K) * K;
        for (int rd = warp; rd < rounds; rd += NT / 32) {
            const int q = (rd / K) * 32 * K + lane * K + rd % K;
            if (q >= len) continue;
            const int p = p0 + q;
            const float4 R = sp.pos[p];
            const int cell = __float_as_int(R.w);
            if (cell < 0) continue;
            int rel[3];
            if (!in_region(cell, rel)) {
                atomicOr(&s_mark[PASSES - 1][q >> 5], 1u << (q & 31));
                continue;
            }
            float4 mo = sp.mom[p];
            const float o[3] = {R.x, R.y, R.z};
            int c[3] = {g.cc.i(cell), g.cc.j(cell), g.cc.k(cell)}, s[3];
            SmemAcc<Reg> acc{reg, sF, sJlo, sJhi, s_js, rel[2] * R2 + rel[1] * Rx + rel[0]};
            float d[3], o1[3], v[3];
            if (!push_move<ORDER, false, 7, SmemAcc<Reg>, GATHER>(acc, o, c, mo, sp, g, ext, err, d, s, o1, zb, v)) {
                sp.pos[p].w = __int_as_float(-1);
                continue;
            }
            sp.mom[p] = mo;
            const bool fits = fabsf(d[0]) <= s_dl[0] && fabsf(d[1]) <= s_dl[1] && fabsf(d[2]) <= s_dl[2];
            if (!fits || !stays_all<ORDER>(o, d, s)) {
                const int oct = (o[0] >= 0.5f) | ((o[1] >= 0.5f) << 1) | ((o[2] >= 0.5f) << 2);
                const int pass = NEUTRAL ? 2 * (oct % gq) / gq : 0;
                atomicOr(&s_mark[pass][q >> 5], 1u << (q & 31));   // its position is still the old one
                continue;
            }
            sp.pos[p] = make_float4(o1[0], o1[1], o1[2], __int_as_float(g.cc.pack(c[0], c[1], c[2])));
#pragma unroll
            for (int k = 0; k < 3; k++) dmax[k] = max(dmax[k], __float_as_uint(fabsf(d[k])));
            const float fac[3] = {sp.cf[0] * mo.w, sp.cf[1] * mo.w, sp.cf[2] * mo.w};
            deposit_simple<ORDER>(acc, o, d, fac);
        }
        __syncthreads();
        // ---- listed records
#pragma unroll
        for (int pass = 0; pass < PASSES; pass++) {
            for (int w = warp; w < (len + 31) / 32; w += NT / 32) {
                const unsigned m = s_mark[pass][w];
                if (m == 0u) continue;
                int at = 0;
                if (lane == 0) at = atomicAdd(&s_n, __popc(m));
                at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
                if ((m >> lane) & 1u) list[at] = (unsigned short)(w * 32 + lane);
            }
            __syncthreads();
        }
        const int n_list = s_n;
        for (int q = tid; q < n_list; q += NT) {
            const int p = p0 + list[q];
            float4 R = sp.pos[p], mo = sp.mom[p];
            int rel[3];
            if (!in_region(__float_as_int(R.w), rel)) {
                step_record<ORDER, false, false, GATHER>(R, mo, sp, g, f, ext, err, dmax);
                sp.mom[p] = mo;
                sp.pos[p] = R;
                continue;
            }
            const int cl = __float_as_int(R.w);
            int c[3] = {g.cc.i(cl), g.cc.j(cl), g.cc.k(cl)}, s[3];
            const int c0[3] = {c[0], c[1], c[2]};
            const float o[3] = {R.x, R.y, R.z};
            float d[3], o1[3], v[3], h[3] = {g.dt_over_d[0], g.dt_over_d[1], g.dt_over_d[2]};
            if (!move<7>(o, c, mo, g, err, d, s, o1, zb, v)) {   // (as in the first loop, which lists none that leaves)
                sp.pos[p].w = __int_as_float(-1);
                continue;
            }
            sp.pos[p] = make_float4(o1[0], o1[1], o1[2], __int_as_float(g.cc.pack(c[0], c[1], c[2])));
            const float fac[3] = {sp.cf[0] * mo.w, sp.cf[1] * mo.w, sp.cf[2] * mo.w};
            const bool fits = fabsf(d[0]) <= s_dl[0] && fabsf(d[1]) <= s_dl[1] && fabsf(d[2]) <= s_dl[2];
            if (!NEUTRAL || q < kQueue)
#pragma unroll
                for (int k = 0; k < 3; k++) { v[k] = d[k]; h[k] = 1.f; }
            bool in = fits;
            int e = 0, crossed = 0;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                dmax[k] = max(dmax[k], __float_as_uint(fabsf(d[k])));
                if (S::stays(o[k], d[k], s[k])) continue;
                e = k;
                crossed++;
                const int st = rel[k] + general_start<ORDER>(o[k], d[k], s[k]);
                in = in && st >= 0 && st + S::L <= (k == 0 ? Rx : (k == 1 ? Ry : Rz));
            }
            if (in && crossed == 1) {
                const SmemAcc<Reg> acc{reg, sF, sJlo, sJhi, s_js, rel[2] * R2 + rel[1] * Rx + rel[0]};
                deposit_cross<ORDER>(acc, o, d, s, fac, e, v, h);
                continue;
            }
            // several dims (its window's tests need every dim), beyond the range or the region
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const int st = rel[k] + general_start<ORDER>(o[k], d[k], s[k]);
                in = in && st >= 0 && st + S::L <= (k == 0 ? Rx : (k == 1 ? Ry : Rz));
            }
            if (in) {
                SmemAcc<Reg> acc{reg, sF, sJlo, sJhi, s_js, rel[2] * R2 + rel[1] * Rx + rel[0]};
                deposit_general<ORDER>(acc, o, d, s, fac, v, h);
            } else {
                GlobAcc<ORDER> acc(f, g, c0, err, zb);
                deposit_general<ORDER>(acc, o, d, s, fac);
                if (!fits) atomicAdd(sp.nfall, 1ull);
            }
        }
        __syncthreads();
        // one flush of the item's current to global memory: hi 2^19 + lo back to float
        const float jinv[3] = {s_jinv[0], s_jinv[1], s_jinv[2]};
        for (int l = tid; l < R3; l += NT) {
            unsigned lo[3];
            int hi[3];
            bool have = false;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                lo[c] = sJlo[c * R3 + l];
                hi[c] = sJhi[c * R3 + l];
                have = have || lo[c] != 0u || hi[c] != 0;
            }
            if (!have) continue;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                sJlo[c * R3 + l] = 0u;
                sJhi[c * R3 + l] = 0;
            }
            const long long gi = node(l);
            if (gi < 0) { atomicOr(err, ERR_INDEX); continue; }   // (plane padding is never written)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                if (lo[c] == 0u && hi[c] == 0) continue;
                const float v = fmaf((float)hi[c], (float)(1u << kLoBits), __uint2float_rn(lo[c])) * jinv[c];
                atomicAdd(f.J + c * g.ncell + gi, v);
            }
        }
    }
    // the step's largest displacement per component (sets the next step's bound)
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const unsigned m = __reduce_max_sync(0xffffffffu, dmax[k]);
        if (lane == 0 && m) atomicMax(sp.dmax + k, m);
    }
    // appended particles not yet sorted, then sparse tiles (fewer than kSparse particles, a warp
    // each): staging and flushing a region would cost more than the global path of these few
    for (int p = n_sorted + blockIdx.x * NT + tid; p < n_total; p += gridDim.x * NT)
        step_global<ORDER, false, false, GATHER>(sp, g, f, ext, err, p);
    const int n_sparse = sp.count[3];
    for (;;) {
        int it = 0;
        if (lane == 0) it = atomicAdd(work_sparse, 1);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= n_sparse) break;
        const int tile = t.sparse_tiles[it];
        const int pe = t.tile_start[tile + 1];
        for (int p = t.tile_start[tile] + lane; p < pe; p += 32) step_global<ORDER, false, true, GATHER>(sp, g, f, ext, err, p);
    }
}

// Plane pitch of the region: rows of a plane's x, the planes 8 (mod 16) words apart, so that the 8 x 4
// cells of a warp in a full tile sit on 32 banks.
__host__ __device__ constexpr int push_pitch(int rx, int ry) { return rx * ry + (24 - (rx * ry) % 16) % 16; }

inline size_t push_smem(int R3) { return (size_t)24 * R3 + std::max((size_t)24 * R3, 2 * (size_t)kChunk); }   // words; fields or list

// Steps since the species' last sort.
inline int sort_age(const pic_ctx *c) { return (int)((c->step - c->sort_base) % c->sort_every); }

template <int ORDER, int GATHER, int NT, int MINB, bool NEUTRAL = false, bool INORDER = false, class Reg>
cudaError_t launch_push_t(pic_ctx *c, int si, const ExtDev &ext, Reg reg, int R3)
{
    static KernelCache cache;
    const Species &s = c->sp[si];
    const size_t smem = push_smem(R3);
    auto kern = k_push<ORDER, GATHER, NT, MINB, NEUTRAL, INORDER, Reg>;
    int per_sm = 0;
    cudaError_t e = cache.blocks_per_sm((const void *)kern, c->dev.device, NT, smem, &per_sm);
    if (e != cudaSuccess) return e;
    kern<<<c->num_sms * std::min(per_sm, MINB), NT, smem, c->stream>>>(species_dev(c, s), grid_dev(c), tile_dev(c, s), FieldsDev{c->E, c->B, c->J},
                                                        ext, c->work + si, c->work + kMaxSpecies + si, c->err, reg, sort_age(c));
    c->kernels++;
    return cudaGetLastError();
}

// The region of a tile: its cells and drift margin, one node below and (TSC) two or (CIC) one above.
template <int ORDER, int GATHER> cudaError_t launch_push_fixed(pic_ctx *c, int si, const ExtDev &ext)
{
    constexpr int R = 8 + 2 * 1 + (ORDER == 1 ? 2 : 3), R2 = push_pitch(R, R);
    // Large species: 2 x 512 threads at 64 registers, whose warps hide more latency than their spills
    // cost.  Small ones, an item or two per CTA, end with their longest thread: 2 x 256 at 128 (300k
    // electrons 0.100 against 0.112 ms per step, 500k 0.115 / 0.130, 3.4M plasma 0.350 / 0.343).
    // (A current that another one nearly cancels: one CTA of 512 at 128 registers, see INORDER.)
    const RegFix<R, R, R, R2> reg;
    if (cancels(c, si)) return launch_push_t<ORDER, GATHER, 512, 1, true, true>(c, si, ext, reg, R2 * R);
    if (c->sp[si].bound <= 8192 * (int64_t)c->num_sms) return launch_push_t<ORDER, GATHER, 256, 2>(c, si, ext, reg, R2 * R);
    return launch_push_t<ORDER, GATHER, 512, 2>(c, si, ext, reg, R2 * R);
}

template <int ORDER, int GATHER> cudaError_t launch_push_dyn(pic_ctx *c, int si, const ExtDev &ext)
{
    int R[3];
    for (int d = 0; d < 3; d++) R[d] = c->T[d] + 2 * c->M + (ORDER == 1 ? 2 : 3);
    const int R2 = push_pitch(R[0], R[1]), R3 = R2 * R[2];
    const RegDyn reg{R[0], R[1], R2, R3};
    // as many CTAs as the region lets on an SM, 512 threads in all
    const size_t cta = push_smem(R3) + 1024 + 768, sm = 228 * 1024;   // with the reserved and the static part
    // A current that another one nearly cancels: one CTA an SM (see INORDER; 2-D buncher, 8 x 1 x 8 tiles:
    // 1.75 ms per step against 1.18 with four CTAs, with a fourth of the scatter of B between launches).  On
    // a 2-D grid, whose tiles have half the neighbours, an item claimed ahead does not add to it (1.97 -> 1.75).
    if (cancels(c, si) && c->n[1] > 1) return launch_push_t<ORDER, GATHER, 512, 1, true, true>(c, si, ext, reg, R3);
    if (cancels(c, si)) return launch_push_t<ORDER, GATHER, 512, 1, true>(c, si, ext, reg, R3);
    if (4 * cta <= sm) return launch_push_t<ORDER, GATHER, 128, 4>(c, si, ext, reg, R3);
    if (2 * cta <= sm) return launch_push_t<ORDER, GATHER, 256, 2>(c, si, ext, reg, R3);
    return launch_push_t<ORDER, GATHER, 512, 1>(c, si, ext, reg, R3);
}

}  // namespace push
}  // namespace gbpic
