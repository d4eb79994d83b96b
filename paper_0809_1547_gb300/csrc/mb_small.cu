// Steps of a small grid: one cooperative launch advances any number of steps,
// the whole state held in the blocks' shared memory.
//
// A block owns a box of tx x ty x tz cells (at most one block per SM).  It
// keeps E with a one-cell halo on every side, H with a halo on the low sides,
// P, J, the populations, 1/eps_r and the CPML memories of its cells; H and
// the psi_H memories of the low halo it advances itself, redundantly (the
// same operations on the same values as their owner, bit for bit), so a step
// exchanges only E: each block writes its boundary cells' E^{n+1} to one half
// of an exchange buffer (the halves used in turn), publishes a step flag and
// waits for the flags of the twelve blocks whose cells its halo holds.
// The gain cells' Lorentz / Langevin update needs own cells only and runs
// between publishing and waiting.
//
// Why: below about 70^3 cells a step is a few microseconds of launches and
// dependent latencies (two field launches and a probe launch: 11.7 us a step
// at 48^3, of which the cells' bytes account for 1.5 us).  Neighbour flags
// instead of a grid barrier: a release store and an acquire load per hop
// instead of two rounds of atomics on one word, and blocks need not run in
// lockstep.  Two halves suffice: a block writes E^{n+2} only after the blocks
// that read its E^n have published E^{n+1}, and the twelve directions are
// closed under negation.
//
// Every update uses the per-cell helpers' operations, so the fields equal
// those of the other launches bit for bit.
//
// Only one such launch fits the GPU at a time (its blocks take nearly all of an
// SM's shared memory): a batch of small grids tries it with all members running.
//
// Measured, per step with a point probe: 24 x 22 x 20 cells 3.1 us, 48^3 4.6
// us (two passes and the probe's launch, tuned: 8.0 and 11.7), plus 10 and 16
// us per launch to load and store the state; the tuner times both parts and
// keeps calls too short to repay the second on the two passes.  What bounds
// it: at 24^3 the chain of a step's latencies (release and acquire of the
// flags about 0.8 us, halo loads 0.4, H 0.4, E 0.7), at 48^3 the instruction
// issue of 24 warps in the same phase (H 0.8, E 1.2).  On the way: flags in
// shared lines cost 1.5 us a step more, FP64 flux sums in the loop 1.2.
#include "mb_host.h"
#include "mb_tiles.cuh"

#include <algorithm>

namespace mb {

namespace {

constexpr int kSmallThreads = 1024;
constexpr int kSmallSpin = 1 << 20;          // polls before a wait gives up (~0.5 s)
constexpr size_t kSmallSmem = 220 * 1024;

// Places (in 16-byte words) of a block's arrays for a box of tx x ty x tz
// cells.  Vectors throughout: a component at a time would cost three times
// the shared-memory instructions and address arithmetic, which bound a step
// here (one or two cells per thread, every warp in the same phase).
struct SmallLayout {
    int e, h, pie, jn, n12, psh, pse, coef, items, halo, total;
    __host__ __device__ SmallLayout(int tx, int ty, int tz, bool pml) {
        const int nc = tx * ty * tz, ne = (tx + 2) * (ty + 2) * (tz + 2), nh = (tx + 1) * (ty + 1) * (tz + 1);
        const int fl = tx * ty + tx * tz + ty * tz;
        e = 0;                                          // float4 (Ex, Ey, Ez, -), halo on every side
        h = e + ne;                                     // float4 (Hx, Hy, Hz, -), halo on the low sides
        pie = h + nh;                                   // float4 (P, 1/eps_r, negative in gain cells)
        jn = pie + nc;                                  // float4 (J, n3)
        n12 = jn + nc;                                  // float2 (n1, n2)
        psh = n12 + (nc + 1) / 2;                       // float2 x 3 axes: psi_H (x: y z, y: x z, z: x y)
        pse = psh + (pml ? (3 * nh + 1) / 2 : 0);       // float2 x 3 axes: psi_E
        coef = pse + (pml ? (3 * nc + 1) / 2 : 0);      // float2 (b, c) per position, E then H, per axis
        items = coef + (pml ? tx + ty + tz + 3 : 0);    // uint2 (place, flags)
        halo = items + (nc + fl + 1) / 2;               // uint2 (place, source)
        total = halo + (2 * fl + 2 * (tx + ty + tz) + 1) / 2;
    }
};

__device__ __forceinline__ unsigned ld_acquire(const unsigned* p) {
    unsigned v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void st_release(unsigned* p, unsigned v) {
    asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Waits (bounded) until the flag has reached `want` (modulo 2^32).
__device__ bool wait_flag(const unsigned* p, unsigned want) {
    for (int it = 0; it < kSmallSpin; ++it)
        if ((int)(ld_acquire(p) - want) >= 0) return true;
    return false;
}

// What is special about a cell (fixed for the launch), found once.
enum : uint32_t {
    kInX = 1, kInY = 2, kInZ = 4,          // lies in a CPML slab
    kEdge = 8,                             // its E is read by other blocks
    kPecX = 16, kPecY = 32, kPecZ = 64,    // Ex / Ey / Ez held at zero
    kFace = 128,                           // may hold face-flux terms
    kSrc = 256,                            // the source cell
    kProbe = 512                           // << p: the cell of probe p
};

// The probes' DFTs: one block per probe, following the owner of its cell
// through the samples that it publishes; running sums in registers, added in
// step order as by k_point_dft.
__device__ void small_probe(const SmallArgs& A, int p, unsigned base, long long n0, int* fail_s) {
    const DevPointProbes& pp = A.pp;
    const int64_t cell = pp.cell[p];
    const int px = A.a.g.px, ny = A.a.g.ny;
    const int gi = (int)(cell % px), gj = (int)(cell / px % ny), gk = (int)(cell / ((int64_t)px * ny));
    const int owner = gi / A.t.tx + A.t.bx * (gj / A.t.ty + A.t.by * (gk / A.t.tz));
    const int K = pp.nfreq, kk = threadIdx.x;
    double2 v[3];
    double w = 0.0;
    if (kk < K) {
        w = pp.omega[p * K + kk];
        for (int c = 0; c < 3; ++c) v[c] = pp.acc[((int64_t)p * 3 + c) * K + kk];
    }
    for (int s = 0; s < A.nsteps; ++s) {
        // the barrier carries the verdict: a flag in shared memory could be set
        // for step s + 1 while a slower warp still reads it for step s
        const bool late = threadIdx.x == 0 && !wait_flag(A.flags + kSmallFlagStride * owner, base + s + 1);
        if (__syncthreads_or(late)) {
            if (late) *fail_s = 1;
            break;
        }
        if (kk < K) {
            const float* e = A.samples + ((size_t)s * pp.count + p) * 3;
            const float2 ph = phase_f32(w, (double)(n0 + s + 1) * A.dt);
            for (int c = 0; c < 3; ++c) {
                const double x = (double)__ldcg(e + c);
                v[c].x += x * (double)ph.x;
                v[c].y += x * (double)ph.y;
            }
        }
    }
    if (kk < K)
        for (int c = 0; c < 3; ++c) pp.acc[((int64_t)p * 3 + c) * K + kk] = v[c];
}

__global__ void __launch_bounds__(kSmallThreads, 1) k_step_small(const __grid_constant__ SmallArgs A) {
    extern __shared__ float4 sm[];
    __shared__ int fail_s;
    __shared__ float3 flux_s[6][kSmallThreads / 32];   // per-warp face-flux sums (add_expansion)
    __shared__ uint32_t pcell[kSmallMaxProbes];
    const StepArgs& a = A.a;
    const DevFields& f = a.f;
    const int T = blockDim.x, tid = threadIdx.x;
    const long long n0 = a.step_ctr[0];
    const unsigned base = *A.base;
    const int nblk = A.t.bx * A.t.by * A.t.bz;
    if (tid == 0) fail_s = 0;
    for (int q = tid; q < 6 * (kSmallThreads / 32); q += T) (&flux_s[0][0])[q] = make_float3(0.f, 0.f, 0.f);
    if (tid < A.pp.count) pcell[tid] = (uint32_t)A.pp.cell[tid];
    __syncthreads();
    if ((int)blockIdx.x >= nblk) {
        small_probe(A, blockIdx.x - nblk, base, n0, &fail_s);
    } else {
        const int bi = blockIdx.x % A.t.bx, bj = blockIdx.x / A.t.bx % A.t.by, bk = blockIdx.x / (A.t.bx * A.t.by);
        const int x0 = bi * A.t.tx, y0 = bj * A.t.ty, z0 = bk * A.t.tz;
        const int nx = a.g.nx, ny = a.g.ny, nz = a.g.nz, L = a.pml.L, L2 = 2 * L;
        const uint32_t nxy = a.g.nxy;
        const int lx = min(A.t.tx, nx - x0), ly = min(A.t.ty, ny - y0), lz = min(A.t.tz, nz - z0);
        const int nc = lx * ly * lz;
        const SmallLayout lay(A.t.tx, A.t.ty, A.t.tz, L > 0);
        // strides of the E and H arrays (own cell (0, 0, 0) at eo, ho)
        const int ey_ = lx + 2, ez_ = ey_ * (ly + 2), NE = ez_ * (lz + 2), eo = 1 + ey_ + ez_;
        const int hy_ = lx + 1, hz_ = hy_ * (ly + 1), NH = hz_ * (lz + 1), ho = 1 + hy_ + hz_;
        float4* const Es = sm + lay.e;
        float4* const Hs = sm + lay.h;
        float4* const Ps = sm + lay.pie;
        float4* const Js = sm + lay.jn;
        float2* const Ns = reinterpret_cast<float2*>(sm + lay.n12);
        float2* const psh = reinterpret_cast<float2*>(sm + lay.psh);
        float2* const pse = reinterpret_cast<float2*>(sm + lay.pse);
        // CPML (b, c) of positions -1 .. l-1 per axis, E sites then H sites
        float2* const cfx = reinterpret_cast<float2*>(sm + lay.coef);
        float2* const cfy = cfx + 2 * (lx + 1);
        float2* const cfz = cfy + 2 * (ly + 1);
        uint2* const items = reinterpret_cast<uint2*>(sm + lay.items);
        uint2* const halo = reinterpret_cast<uint2*>(sm + lay.halo);

        // which slabs a position lies in, and the places of its CPML memories
        auto in_x = [&](int gi) { return L > 0 && (gi < L || gi >= nx - L); };
        auto in_y = [&](int gj) { return L > 0 && (gj < L || gj >= ny - L); };
        auto in_z = [&](int gk) { return L > 0 && (gk < a.pml.zlo || gk >= a.pml.zhi); };
        const uint32_t plx = (uint32_t)nz * ny * L2, ply = (uint32_t)nz * L2 * nx, plz = (uint32_t)a.pml.zn * ny * nx;
        auto qx = [&](int gi, int gj, int gk) { return ((uint32_t)gk * ny + gj) * L2 + slab_index(gi, nx, L); };
        auto qy = [&](int gi, int gj, int gk) { return ((uint32_t)gk * L2 + slab_index(gj, ny, L)) * nx + gi; };
        auto qz = [&](int gi, int gj, int gk) {
            const uint32_t s = gk < a.pml.zlo ? gk : gk - a.pml.zhi + a.pml.zs;
            return (s * ny + gj) * nx + gi;
        };

        for (int q = tid; q < NE; q += T) Es[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = tid; q < NH; q += T) Hs[q] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (L > 0) {
            const float* tab[3][4] = {{a.pml.bex, a.pml.cex, a.pml.bhx, a.pml.chx},
                                      {a.pml.bey, a.pml.cey, a.pml.bhy, a.pml.chy},
                                      {a.pml.bez, a.pml.cez, a.pml.bhz, a.pml.chz}};
            float2* dst = cfx;
#pragma unroll
            for (int w = 0; w < 3; ++w) {
                const int l = w == 0 ? lx : w == 1 ? ly : lz, o = w == 0 ? x0 : w == 1 ? y0 : z0;
#pragma unroll
                for (int c = 0; c < 2; ++c)
                    for (int q = tid; q <= l; q += T)
                        if (o + q >= 1)
                            dst[c * (l + 1) + q] = make_float2(__ldg(tab[w][2 * c] + o + q - 1),
                                                               __ldg(tab[w][2 * c + 1] + o + q - 1));
                dst += 2 * (l + 1);
            }
        }
        __syncthreads();   // (the zeros before the values)

        // ---- own cells and low-side halo cells: place (i+1, j+1, k+1),
        // flags and the state at n0
        const int hx = x0 > 0 ? ly * lz : 0, hyn = y0 > 0 ? lx * lz : 0, hzn = z0 > 0 ? lx * ly : 0;
        const int nitems = nc + hx + hyn + hzn;
        for (int q = tid; q < nitems; q += T) {
            int i, j, k, r = q;
            if (r < nc) {
                i = r % lx; j = r / lx % ly; k = r / (lx * ly);
            } else if ((r -= nc) < hx) {
                i = -1; j = r % ly; k = r / ly;
            } else if ((r -= hx) < hyn) {
                i = r % lx; j = -1; k = r / lx;
            } else {
                r -= hyn;
                i = r % lx; j = r / lx; k = -1;
            }
            const int gi = x0 + i, gj = y0 + j, gk = z0 + k;
            const uint32_t c = cell_place(a.g, gi, gj, gk);
            const int hp = ho + i + hy_ * j + hz_ * k;
            Hs[hp] = make_float4(f.hx[c], f.hy[c], f.hz[c], 0.f);
            uint32_t fl = 0;
            if (in_x(gi)) {
                const uint32_t p = qx(gi, gj, gk);
                fl |= kInX;
                psh[hp] = make_float2(a.pml.psx[p + 2 * plx], a.pml.psx[p + 3 * plx]);
                if (q < nc) pse[q] = make_float2(a.pml.psx[p], a.pml.psx[p + plx]);
            }
            if (in_y(gj)) {
                const uint32_t p = qy(gi, gj, gk);
                fl |= kInY;
                psh[NH + hp] = make_float2(a.pml.psy[p + 2 * ply], a.pml.psy[p + 3 * ply]);
                if (q < nc) pse[nc + q] = make_float2(a.pml.psy[p], a.pml.psy[p + ply]);
            }
            if (in_z(gk)) {
                const uint32_t p = qz(gi, gj, gk);
                fl |= kInZ;
                psh[2 * NH + hp] = make_float2(a.pml.psz[p + 2 * plz], a.pml.psz[p + 3 * plz]);
                if (q < nc) pse[2 * nc + q] = make_float2(a.pml.psz[p], a.pml.psz[p + plz]);
            }
            if (q < nc) {
                if (i == 0 || j == 0 || k == 0 || i == lx - 1 || j == ly - 1 || k == lz - 1) fl |= kEdge;
                if (gj == 0 || gk == 0) fl |= kPecX;
                if (gi == 0 || gk == 0) fl |= kPecY;
                if (gi == 0 || gj == 0) fl |= kPecZ;
                if (a.flux.on && (cells_on_xy_face(a.flux, gi, 1, gj) || gk == a.flux.plo[2] || gk == a.flux.phi[2]))
                    fl |= kFace;
                if (a.src.on && c == (uint32_t)a.src.cell) fl |= kSrc;
                for (int p = 0; p < A.pp.count; ++p)
                    if (pcell[p] == c) fl |= kProbe << p;
                Es[eo + i + ey_ * j + ez_ * k] = make_float4(f.ex[c], f.ey[c], f.ez[c], 0.f);
                const uint8_t m = f.mat[c];
                const float ie = f.inv_eps ? f.inv_eps[c] : f.lut_inv_eps[m & 0x7f];
                const bool g = a.gain.on && (m & 0x80);
                const float* gs = f.gs + gain_place(c);
                Ps[q] = make_float4(gs[kPx], gs[kPy], gs[kPz], g ? -ie : ie);
                Js[q] = make_float4(gs[kJx], gs[kJy], gs[kJz], gs[kN3]);
                Ns[q] = make_float2(gs[kN1], gs[kN2]);
            }
            items[q] = make_uint2((uint32_t)(i + 1) | (uint32_t)(j + 1) << 10 | (uint32_t)(k + 1) << 20, fl);
        }
        // ---- halo cells of E: place and source (an entry of the exchange
        // buffer: the owner's block and its cell's number there)
        const int ncmax = A.t.tx * A.t.ty * A.t.tz;
        const int fx = ly * lz, fy = lx * lz, fz = lx * ly;
        const int nhalo = 2 * (fx + fy + fz) + 2 * (lx + ly + lz);
        for (int q = tid; q < nhalo; q += T) {
            int i, j, k, r = q;
            if (r < 2 * fx) { i = r < fx ? -1 : lx; r %= fx; j = r % ly; k = r / ly; }
            else if ((r -= 2 * fx) < 2 * fy) { j = r < fy ? -1 : ly; r %= fy; i = r % lx; k = r / lx; }
            else if ((r -= 2 * fy) < 2 * fz) { k = r < fz ? -1 : lz; r %= fz; i = r % lx; j = r / lx; }
            else if ((r -= 2 * fz) < 2 * lz) { i = r < lz ? -1 : lx; j = r < lz ? ly : -1; k = r % lz; }
            else if ((r -= 2 * lz) < 2 * ly) { i = r < ly ? -1 : lx; k = r < ly ? lz : -1; j = r % ly; }
            else { r -= 2 * ly; j = r < lx ? -1 : ly; k = r < lx ? lz : -1; i = r % lx; }
            const int gi = x0 + i, gj = y0 + j, gk = z0 + k;
            const int ep = eo + i + ey_ * j + ez_ * k;
            uint32_t src = 0xffffffffu;
            if (gi >= 0 && gi < nx && gj >= 0 && gj < ny && gk >= 0 && gk < nz) {
                const uint32_t c = cell_place(a.g, gi, gj, gk);
                Es[ep] = make_float4(f.ex[c], f.ey[c], f.ez[c], 0.f);
                const int ob = gi / A.t.tx, oj = gj / A.t.ty, ok = gk / A.t.tz;
                const int olx = min(A.t.tx, nx - ob * A.t.tx), oly = min(A.t.ty, ny - oj * A.t.ty);
                src = (uint32_t)((ob + A.t.bx * (oj + A.t.by * ok)) * ncmax + (gi - ob * A.t.tx) +
                                 olx * ((gj - oj * A.t.ty) + oly * (gk - ok * A.t.tz)));
            }
            halo[q] = make_uint2((uint32_t)ep, src);
        }
        // the flag this lane of the last warp waits for: the neighbour in one of
        // the twelve directions that the halo of E reaches (the last warp
        // publishes and waits: it holds few own cells or none, so the others'
        // flux sums and Lorentz update run meanwhile)
        const int svc = tid - (T - 32);
        int nbr = -1;
        if (svc >= 0 && svc < 12) {
            const int dxs[12] = {-1, 1, 0, 0, 0, 0, -1, 1, -1, 1, 0, 0};
            const int dys[12] = {0, 0, -1, 1, 0, 0, 1, -1, 0, 0, -1, 1};
            const int dzs[12] = {0, 0, 0, 0, -1, 1, 0, 0, 1, -1, 1, -1};
            const int i = bi + dxs[svc], j = bj + dys[svc], k = bk + dzs[svc];
            if (i >= 0 && i < A.t.bx && j >= 0 && j < A.t.by && k >= 0 && k < A.t.bz)
                nbr = i + A.t.bx * (j + A.t.by * k);
        }
        const bool face = tile_on_face(a.flux, x0, x0 + lx, y0, y0 + ly, z0, z0 + lz);
        __syncthreads();

        // the thread's first item, kept in registers (most boxes have no more
        // items than threads)
        struct Item {
            int ep, hp;         // places in E and H
            uint32_t pos, fl;   // (i+1, j+1, k+1), flags
        };
        auto decode = [&](int q) {
            const uint2 v = items[q];
            const int i = (int)(v.x & 1023u) - 1, j = (int)(v.x >> 10 & 1023u) - 1, k = (int)(v.x >> 20) - 1;
            return Item{eo + i + ey_ * j + ez_ * k, ho + i + hy_ * j + hz_ * k, v.x, v.y};
        };
        const Item first = decode(min(tid, nitems - 1));
        auto item = [&](int q) { return q == tid ? first : decode(q); };
        auto cell = [&](uint32_t pos) {
            return cell_place(a.g, x0 - 1 + (int)(pos & 1023u), y0 - 1 + (int)(pos >> 10 & 1023u), z0 - 1 + (int)(pos >> 20));
        };
        // J^{n+1/2}, P^{n+1} of the own gain cells (time-n values of own cells only)
        auto lorentz = [&](long long n) {
            for (int q = tid; q < nc; q += T) {
                float4 p = Ps[q];
                if (!(p.w < 0.0f)) continue;
                const Item m = item(q);
                const float4 e = Es[m.ep];
                float4 j = Js[q];
                const float2 nn = Ns[q];
                lorentz_step(a.gain, cell_number(a.g, x0 - 1 + (int)(m.pos & 1023u), y0 - 1 + (int)(m.pos >> 10 & 1023u),
                                                 z0 - 1 + (int)(m.pos >> 20)),
                             n, e.x, e.y, e.z, nn.x, nn.y, j.x, j.y, j.z, p.x, p.y, p.z);
                Ps[q] = p;
                Js[q] = j;
            }
        };
        if (a.gain.on) lorentz(n0);

        const float S = a.S;
        const size_t half = (size_t)nblk * ncmax;   // the exchange buffer's two halves, used in turn
        for (int s = 0; s < A.nsteps; ++s) {
            const long long n = n0 + s;
            if (s > 0) {
                __syncthreads();   // (the waits below, at the end of the step before)
                if (fail_s) break;
                const float4* x = A.xbuf + (s & 1) * half;
                for (int q = tid; q < nhalo; q += T) {
                    const uint2 h = halo[q];
                    if (h.y != 0xffffffffu) Es[h.x] = __ldcg(x + h.y);
                }
                __syncthreads();
            }
            // 1. H^{n+1/2} of the own cells and of the low-side halo
            for (int q = tid; q < nitems; q += T) {
                const Item m = item(q);
                const float4 e = Es[m.ep], ei = Es[m.ep + 1], ej = Es[m.ep + ey_], ek = Es[m.ep + ez_];
                const float d0 = ej.z - e.z, d1 = ek.y - e.y, d2 = ek.x - e.x;   // dEz_dy, dEy_dz, dEx_dz
                const float d3 = ei.z - e.z, d4 = ei.y - e.y, d5 = ej.x - e.x;   // dEz_dx, dEy_dx, dEx_dy
                float cx = d0 - d1, cy = d2 - d3, cz = d4 - d5;
                if (m.fl & kInX) {
                    const float2 bc = cfx[lx + 1 + (m.pos & 1023u)];
                    float2 u = psh[m.hp];
                    u = make_float2(fmaf(bc.x, u.x, bc.y * d3), fmaf(bc.x, u.y, bc.y * d4));
                    psh[m.hp] = u;
                    cy -= u.x;
                    cz += u.y;
                }
                if (m.fl & kInY) {
                    const float2 bc = cfy[ly + 1 + (m.pos >> 10 & 1023u)];
                    float2 u = psh[NH + m.hp];
                    u = make_float2(fmaf(bc.x, u.x, bc.y * d0), fmaf(bc.x, u.y, bc.y * d5));
                    psh[NH + m.hp] = u;
                    cx += u.x;
                    cz -= u.y;
                }
                if (m.fl & kInZ) {
                    const float2 bc = cfz[lz + 1 + (m.pos >> 20)];
                    float2 u = psh[2 * NH + m.hp];
                    u = make_float2(fmaf(bc.x, u.x, bc.y * d1), fmaf(bc.x, u.y, bc.y * d2));
                    psh[2 * NH + m.hp] = u;
                    cx -= u.x;
                    cy += u.y;
                }
                float4 h = Hs[m.hp];
                h.x = fmaf(-S, cx, h.x);
                h.y = fmaf(-S, cy, h.y);
                h.z = fmaf(-S, cz, h.z);
                Hs[m.hp] = h;
            }
            __syncthreads();
            // 2. E^{n+1}, N^{n+1}, face flux; the boundary cells' E published
            const bool last = s + 1 == A.nsteps;
            float4* const xo = A.xbuf + ((s + 1) & 1) * half + (size_t)blockIdx.x * ncmax;
            float fl[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            bool on_face = false;
            for (int q = tid; q < nc; q += T) {
                const Item m = item(q);
                const float4 h0 = Hs[m.hp], hi = Hs[m.hp - 1], hj = Hs[m.hp - hy_], hk = Hs[m.hp - hz_];
                const HNb h{h0.x, h0.y, h0.z, hj.x, hk.x, hi.y, hk.y, hi.z, hj.z};
                const float d0 = h.hz - h.hz_j, d1 = h.hy - h.hy_k, d2 = h.hx - h.hx_k;
                const float d3 = h.hz - h.hz_i, d4 = h.hy - h.hy_i, d5 = h.hx - h.hx_j;
                float cx = d0 - d1, cy = d2 - d3, cz = d4 - d5;
                if (m.fl & kInX) {
                    const float2 bc = cfx[m.pos & 1023u];
                    float2 u = pse[q];
                    u = make_float2(fmaf(bc.x, u.x, bc.y * d3), fmaf(bc.x, u.y, bc.y * d4));
                    pse[q] = u;
                    cy -= u.x;
                    cz += u.y;
                }
                if (m.fl & kInY) {
                    const float2 bc = cfy[m.pos >> 10 & 1023u];
                    float2 u = pse[nc + q];
                    u = make_float2(fmaf(bc.x, u.x, bc.y * d0), fmaf(bc.x, u.y, bc.y * d5));
                    pse[nc + q] = u;
                    cx += u.x;
                    cz -= u.y;
                }
                if (m.fl & kInZ) {
                    const float2 bc = cfz[m.pos >> 20];
                    float2 u = pse[2 * nc + q];
                    u = make_float2(fmaf(bc.x, u.x, bc.y * d1), fmaf(bc.x, u.y, bc.y * d2));
                    pse[2 * nc + q] = u;
                    cx -= u.x;
                    cy += u.y;
                }
                const float iv = Ps[q].w;
                const bool g = iv < 0.0f;
                const float ie = fabsf(iv);
                float4 j4 = make_float4(0.f, 0.f, 0.f, 0.f);
                if (g) j4 = Js[q];
                float sx = j4.x, sy = j4.y, sz = j4.z;
                if (m.fl & kSrc) {
                    const float v = source_value(a.src, n);
                    if (a.src.comp == 0) sx += v;
                    else if (a.src.comp == 1) sy += v;
                    else sz += v;
                }
                const float4 e = Es[m.ep];
                float ex1 = fmaf(ie, fmaf(S, cx, -sx), e.x);
                float ey1 = fmaf(ie, fmaf(S, cy, -sy), e.y);
                float ez1 = fmaf(ie, fmaf(S, cz, -sz), e.z);
                if (m.fl & kPecX) ex1 = 0.0f;
                if (m.fl & kPecY) ey1 = 0.0f;
                if (m.fl & kPecZ) ez1 = 0.0f;
                const float4 e1 = make_float4(ex1, ey1, ez1, 0.f);
                Es[m.ep] = e1;
                if (m.fl & kEdge) xo[q] = e1;
                if (g) {
                    float2 nn = Ns[q];
                    population_step(a.gain, e.x, e.y, e.z, ex1, ey1, ez1, j4.x, j4.y, j4.z, nn.x, nn.y, j4.w);
                    Ns[q] = nn;
                    Js[q].w = j4.w;
                }
                if (m.fl & kFace) {
                    on_face = true;
                    flux_terms(a.flux, x0 - 1 + (int)(m.pos & 1023u), y0 - 1 + (int)(m.pos >> 10 & 1023u),
                               z0 - 1 + (int)(m.pos >> 20), h, e.x, e.y, e.z, ex1, ey1, ez1, fl);
                }
                for (int p = 0; m.fl >= (kProbe << p); ++p)
                    if (m.fl & (kProbe << p)) {
                        float* x = A.samples + ((size_t)s * A.pp.count + p) * 3;
                        x[0] = ex1;
                        x[1] = ey1;
                        x[2] = ez1;
                    }
            }
            __syncthreads();
            if (svc == 31) st_release(A.flags + kSmallFlagStride * blockIdx.x, base + s + 1);   // (cumulative over the barrier)
            if (face && __any_sync(0xffffffffu, on_face)) {
                // face flux, while the flags travel: warp sums, added to the
                // warp's running sums in three FP32 parts, more bits than FP64
                // holds (an FP64 addition costs about a microsecond of latency here)
#pragma unroll
                for (int w = 0; w < 6; ++w) {
                    float v = fl[w];
                    if (__any_sync(0xffffffffu, v != 0.0f)) {
#pragma unroll
                        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
                        if ((tid & 31) == 0) {
                            float3 p = flux_s[w][tid >> 5];
                            add_expansion(v, p.x, p.y, p.z);
                            flux_s[w][tid >> 5] = p;
                        }
                    }
                }
            }
            if (!last && a.gain.on) lorentz(n + 1);
            __syncwarp();
            if (!last && nbr >= 0 && !wait_flag(A.flags + kSmallFlagStride * nbr, base + s + 1)) fail_s = 1;
        }
        __syncthreads();

        // ---- the state at the end: E, H and the CPML memories to the copy
        // that holds it (never the one a neighbour may still be loading from:
        // for one step it is the other copy, for more the neighbours' flags
        // say that they have loaded), the rest in place
        const bool other = A.nsteps & 1;
        float* const out[6] = {other ? A.d.ex : f.ex, other ? A.d.ey : f.ey, other ? A.d.ez : f.ez,
                               other ? A.d.hx : f.hx, other ? A.d.hy : f.hy, other ? A.d.hz : f.hz};
        float* const px_o = other ? A.d.psi.x : a.pml.psx;
        float* const py_o = other ? A.d.psi.y : a.pml.psy;
        float* const pz_o = other ? A.d.psi.z : a.pml.psz;
        for (int q = tid; q < nc; q += T) {
            const Item m = item(q);
            const int gi = x0 - 1 + (int)(m.pos & 1023u), gj = y0 - 1 + (int)(m.pos >> 10 & 1023u),
                      gk = z0 - 1 + (int)(m.pos >> 20);
            const uint32_t c = cell(m.pos);
            const float4 e = Es[m.ep], h = Hs[m.hp], p4 = Ps[q];
            out[0][c] = e.x;
            out[1][c] = e.y;
            out[2][c] = e.z;
            out[3][c] = h.x;
            out[4][c] = h.y;
            out[5][c] = h.z;
            if (p4.w < 0.0f) {
                const float4 j4 = Js[q];
                const float2 nn = Ns[q];
                float* gs = f.gs + gain_place(c);
                gs[kPx] = p4.x;
                gs[kPy] = p4.y;
                gs[kPz] = p4.z;
                gs[kJx] = j4.x;
                gs[kJy] = j4.y;
                gs[kJz] = j4.z;
                gs[kN1] = nn.x;
                gs[kN2] = nn.y;
                gs[kN3] = j4.w;
            }
            if (m.fl & kInX) {
                const uint32_t p = qx(gi, gj, gk);
                px_o[p] = pse[q].x;
                px_o[p + plx] = pse[q].y;
                px_o[p + 2 * plx] = psh[m.hp].x;
                px_o[p + 3 * plx] = psh[m.hp].y;
            }
            if (m.fl & kInY) {
                const uint32_t p = qy(gi, gj, gk);
                py_o[p] = pse[nc + q].x;
                py_o[p + ply] = pse[nc + q].y;
                py_o[p + 2 * ply] = psh[NH + m.hp].x;
                py_o[p + 3 * ply] = psh[NH + m.hp].y;
            }
            if (m.fl & kInZ) {
                const uint32_t p = qz(gi, gj, gk);
                pz_o[p] = pse[2 * nc + q].x;
                pz_o[p + plz] = pse[2 * nc + q].y;
                pz_o[p + 2 * plz] = psh[2 * NH + m.hp].x;
                pz_o[p + 3 * plz] = psh[2 * NH + m.hp].y;
            }
        }
        if (tid < 6) {
            double v = 0.0;
            for (int w = 0; w < (T >> 5); ++w) v += (double)flux_s[tid][w].x + ((double)flux_s[tid][w].y + (double)flux_s[tid][w].z);
            if (v != 0.0) atomicAdd(a.flux.acc + tid * kFluxSlots + blockIdx.x % kFluxSlots, v);
        }
    }
    __syncthreads();
    if (tid == 0) {
        if (fail_s) atomicOr(a.err, 1);
        __threadfence();
        // the last block to finish (every block has read n0 and base)
        if (atomicAdd((unsigned long long*)(a.step_ctr + 1), 1ull) == gridDim.x - 1) {
            a.step_ctr[1] = 0;
            a.step_ctr[0] = n0 + A.nsteps;
            *A.d.sample = n0 + A.nsteps;
            *A.sample_in = n0 + A.nsteps;
            *A.base = base + (unsigned)A.nsteps;
        }
    }
}

}  // namespace

// The box and the number of blocks for a grid: the fewest cells (halo cells
// included, as each costs an H update) in the busiest block among the boxes
// that need at most max_blocks blocks and fit in shared memory.  Fewer cells
// per block means fewer passes of its threads per step; the halo grows as
// boxes shrink.
bool small_tile(const DevGrid& g, bool pml, int max_blocks, SmallTile* out) {
    long best = -1;
    if (max_blocks < 1 || g.nx > 1000 || g.ny > 1000 || g.nz > 1000) return false;
    for (int bz = 1; bz <= std::min(g.nz, max_blocks); ++bz)
        for (int by = 1; by * bz <= max_blocks && by <= g.ny; ++by)
            for (int bx = 1; bx * by * bz <= max_blocks && bx <= g.nx; ++bx) {
                const int tx = (g.nx + bx - 1) / bx, ty = (g.ny + by - 1) / by, tz = (g.nz + bz - 1) / bz;
                // every block owns cells (the last box of an axis is not empty)
                if ((bx - 1) * tx >= g.nx || (by - 1) * ty >= g.ny || (bz - 1) * tz >= g.nz) continue;
                if (sizeof(float4) * (size_t)SmallLayout(tx, ty, tz, pml).total > kSmallSmem) continue;
                const long work = (long)tx * ty * tz + tx * ty + tx * tz + ty * tz;
                if (best < 0 || work < best) {
                    best = work;
                    *out = {tx, ty, tz, bx, by, bz};
                }
            }
    return best >= 0;
}

cudaError_t launch_step_small(const SmallArgs& A, cudaStream_t s) {
    const int smem = (int)sizeof(float4) * SmallLayout(A.t.tx, A.t.ty, A.t.tz, A.a.pml.L > 0).total;
    cudaError_t e = cudaFuncSetAttribute(k_step_small, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallSmem);
    if (e != cudaSuccess) return e;
    const int work = A.t.tx * A.t.ty * A.t.tz + A.t.tx * A.t.ty + A.t.tx * A.t.tz + A.t.ty * A.t.tz;
    // a thread per cell and halo cell where they fit; a probe block needs a thread per bin
    int threads = (work + 31) / 32 * 32;
    if (A.pp.count > 0) threads = std::max(threads, (A.pp.nfreq + 31) / 32 * 32);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(A.t.bx * A.t.by * A.t.bz + A.pp.count, 1, 1);
    cfg.blockDim = dim3(std::min(std::max(threads, 64), kSmallThreads), 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;   // all blocks co-resident: the flag waits are safe
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_step_small, A);
}

}  // namespace mb
