// The fused step on patches: where row marches would be short, where their
// strips fit the lattice badly, for the phase counts and models that run
// faster so at any size (use_patches), and for 16-bit storage.
//
// step_tile marches a strip of columns down the lattice: every row costs one
// round trip to memory and two barriers, and each chunk repeats 4 + 2
// pre-roll rows.  A lattice that does not fill the GPU with long chunks
// spends its time in those (256^2: chunks of 2 rows, 6 rows of latency, each
// node's pull repeated three times).  Here a block owns a patch of PX x PY
// nodes instead and runs the three stages once:
//   A  phi on the patch and a two-node ring around it, pulled straight from
//      global memory (all loads of a node in flight at once); the own nodes
//      keep j and phi_lo;
//   B  grad phi, the source, m_phi and w on the patch and a one-node ring;
//   C  the node is completed (complete_node).
// Only (PX + 4)(PY + 4) / (PX PY) - 1 of the pulls are repeated.  The
// arithmetic of a node is the one of step_tile, operation by operation, so
// the two give the same bits.
#pragma once

namespace nlbm {

// Indices of the nine populations node (x, y) pulls: element idx[i] of a
// phase's [9][plane] array.  inside: the node and its neighbours lie within
// the lattice.
__device__ __forceinline__ void pull_index(const StepParams &P, int x, int y, bool inside, unsigned (&idx)[9])
{
    const unsigned pl = P.plane;
    if (inside) {
        const unsigned nx = (unsigned)P.nx, self = (unsigned)y * nx + x;
#pragma unroll
        for (int i = 0; i < 9; ++i) idx[i] = self + ((unsigned)i * pl - (unsigned)cx_of(i) - (unsigned)cy_of(i) * nx);
    } else {
        unsigned node[9];
        int dir[9];
        pull_sources(P, x, y, node, dir);
#pragma unroll
        for (int i = 0; i < 9; ++i) idx[i] = (unsigned)dir[i] * pl + node[i];
    }
}

// phi (and, for an own node, phi_lo and j) of one node pulled from global
// memory; self is the node.
template <class V, int NS, int ST, bool OWN>
__device__ __forceinline__ void pull_direct_v(const StepParams &P, const unsigned (&idx)[9], unsigned self, int p,
                                              float *ph, float *plo, float *jx, float *jy)
{
    const unsigned pl = P.plane;
    auto ld = [](const float *a, size_t stride, auto tag) {
        using U = decltype(tag);
        if constexpr (sizeof(U) == 8) return make_float2(__ldg(a), __ldg(a + stride));
        else return __ldg(a);
    };
    V f[9];
    if constexpr (ST == 0) {
#pragma unroll
        for (int i = 0; i < 9; ++i) f[i] = ld(P.fin + (size_t)p * 9 * pl + idx[i], (size_t)9 * pl, V());
    } else {
        // idx counts from direction 0; the deviations start at direction 1
        f[0] = ld(P.f0in + (size_t)p * pl + self, pl, V());
        const V own = ld(P.phi_prev + (size_t)p * pl + self, pl, V());
#pragma unroll
        for (int i = 1; i < 9; ++i) {
            V dev;
            if constexpr (sizeof(V) == 8)
                dev = Pack16<ST>::dec2(__ldg((const unsigned *)P.fin + dev_word(p / 2, 0, pl, idx[i] - pl)));
            else
                dev = Store16<ST>::dec(__ldg((const unsigned short *)P.fin + dev_tail(NS, 0, pl, idx[i] - pl)));
            f[i] = vfma(vset<V>(w_of(i)), own, dev);
        }
    }
    V a, lo, x, y;
    pull_moments<V, OWN>(f, a, lo, x, y);
    vput(ph, p, a);
    if (OWN) { vput(plo, p, lo); vput(jx, p, x); vput(jy, p, y); }
}
template <int NS, int ST, bool OWN>
__device__ __forceinline__ void pull_direct(const StepParams &P, const unsigned (&idx)[9], unsigned self,
                                            float (&ph)[NS], float (&plo)[NS], float (&jx)[NS], float (&jy)[NS])
{
#pragma unroll
    for (int p = 0; p + 1 < NS; p += 2) pull_direct_v<float2, NS, ST, OWN>(P, idx, self, p, ph, plo, jx, jy);
    if (NS & 1) pull_direct_v<float, NS, ST, OWN>(P, idx, self, NS - 1, ph, plo, jx, jy);
}

// OwnRing's counterpart: j and phi_lo in the thread's own slots, and phi of a
// neighbour (16-bit storage) in the patch's ring (row of 2 ceil(NS / 2) values
// per column, see ring_idx).
template <int NS, int RX, int T>
struct OwnPatch {
    const float *s_j, *s_phi;   // s_phi: the node's row
    int t, c;                   // thread, ring column
    static constexpr int NE = ring_even(NS);
    template <class V> __device__ __forceinline__ V jx(int p) const { return rld<V>(s_j, T, p, t); }
    template <class V> __device__ __forceinline__ V jy(int p) const { return rld<V>(s_j + NE * T, T, p, t); }
    template <class V> __device__ __forceinline__ V plo(int p) const { return rld<V>(s_j + 2 * NE * T, T, p, t); }
    template <class V> __device__ __forceinline__ V phi_at(int p, int cx, int cy) const
    {
        return rld<V>(s_phi + cy * NE * RX, RX, p, c + cx);
    }
};

template <int NS, int PX, int PY>
constexpr size_t patch_smem_bytes()
{
    return sizeof(float) * ((size_t)(PX + 4) * (PY + 4) * ring_even(NS) + (size_t)(PX + 2) * (PY + 2) +
                            (size_t)3 * ring_even(NS) * PX * PY);
}

template <int NS, int MODEL, int ST, int PX, int PY, bool TAPE = false>
__device__ __forceinline__ void step_patch(const StepParams &P, const int x0, const int y0, float *smem)
{
    constexpr int N = NS + 1, T = PX * PY, RX = PX + 4, RY = PY + 4, BX = PX + 2, NE = ring_even(NS);
    float *s_phi = smem;                    // [RY][NE/2][RX][2]
    float *s_j = s_phi + RX * RY * NE;      // [3][NE/2][T][2] j_x, j_y, phi_lo of the own nodes
    float *s_w = s_j + 3 * NE * T;          // [PY + 2][BX]
    const int t = threadIdx.x, lx = t % PX, ly = t / PX;
    const int We = min(PX, P.nx - x0), He = min(PY, P.ny - y0);
    const unsigned pl = P.plane;
    // every pull of the block's nodes stays within the lattice
    const bool inside = x0 >= 3 && y0 >= 3 && x0 + We + 3 <= P.nx && y0 + He + 3 <= P.ny;
    const bool own = lx < We && ly < He;
    const int x = x0 + lx, y = y0 + ly;
    const unsigned node = (unsigned)y * P.nx + x;

    // ---------------------------------------------------- stage A
    float g[9], php[NS], mpx = 0.f, mpy = 0.f, upx = 0.f, upy = 0.f;
    if (own) {
        unsigned idx[9];
        pull_index(P, x, y, inside, idx);
        float ph[NS], plo[NS], jx[NS], jy[NS];
        pull_direct<NS, ST, true>(P, idx, node, ph, plo, jx, jy);
        float *prow = s_phi + (ly + 2) * NE * RX;
#pragma unroll
        for (int p = 0; p + 1 < NS; p += 2) {
            rst(prow, RX, p, lx + 2, vget<float2>(ph, p));
            rst(s_j, T, p, t, vget<float2>(jx, p));
            rst(s_j + NE * T, T, p, t, vget<float2>(jy, p));
            rst(s_j + 2 * NE * T, T, p, t, vget<float2>(plo, p));
        }
        if (NS & 1) {
            rst(prow, RX, NS - 1, lx + 2, ph[NS - 1]);
            rst(s_j, T, NS - 1, t, jx[NS - 1]);
            rst(s_j + NE * T, T, NS - 1, t, jy[NS - 1]);
            rst(s_j + 2 * NE * T, T, NS - 1, t, plo[NS - 1]);
        }
        // what stages B and C read of this node, requested before the barriers
        upx = __ldg(P.uin + node);
        upy = __ldg(P.uin + pl + node);
        if constexpr (ST == 0) {
#pragma unroll
            for (int i = 1; i < 9; ++i) g[i] = __ldg(P.gin + (idx[i] - pl));
        } else {
            unsigned gnode[9];
            int gdir[9];
            pull_sources(P, x, y, gnode, gdir);
#pragma unroll
            for (int i = 1; i < 9; ++i)
                g[i] = __fmaf_rn(3.f * w_of(i), __ldg(P.pin + gnode[i]),
                                 Store16<ST>::dec(__ldg((const unsigned short *)P.gin + (idx[i] - pl))));
        }
#pragma unroll
        for (int p = 0; p < NS; ++p) php[p] = P.phi_prev[(size_t)p * pl + node];
        mpx = P.mphi_in[node];
        mpy = P.mphi_in[pl + node];
    }
    // the ring: two rows below and above the patch, then two columns beside it
    for (int h = t; h < 4 * RX + 4 * PY; h += T) {
        int rx, ry;   // offset from (x0, y0)
        if (h < 4 * RX) {
            const int r = h / RX;
            rx = h - r * RX - 2;
            ry = r < 2 ? r - 2 : He + r - 2;
        } else {
            const int k = h - 4 * RX;
            ry = k >> 2;
            rx = (k & 3) < 2 ? (k & 3) - 2 : We + (k & 3) - 2;
        }
        if (rx >= We + 2 || (h >= 4 * RX && ry >= He)) continue;
        bool fx, fy;
        const int xc = map_axis(x0 + rx, P.nx, P.wall_x, fx), yc = map_axis(y0 + ry, P.ny, P.wall_y, fy);
        unsigned idx[9];
        pull_index(P, xc, yc, inside, idx);
        float ph[NS], plo[NS], jx[NS], jy[NS];
        pull_direct<NS, ST, false>(P, idx, (unsigned)yc * P.nx + xc, ph, plo, jx, jy);
        if (P.wet && (y0 + ry < 0 || y0 + ry >= P.ny)) wet_ghost<NS>(P, y0 + ry, ph);
        float *prow = s_phi + (ry + 2) * NE * RX;
#pragma unroll
        for (int p = 0; p + 1 < NS; p += 2) rst(prow, RX, p, rx + 2, vget<float2>(ph, p));
        if (NS & 1) rst(prow, RX, NS - 1, rx + 2, ph[NS - 1]);
    }
    __syncthreads();

    // ---------------------------------------------------- stage B
    float Rx[NS], Ry[NS], mx = 0.f, my = 0.f;
    float PH[NS], GX[NS], GY[NS], LP[NS];
    if (own) {
        float ph[N], gx[N], gy[N], lap[N];
        window_grad_lap<NS>(s_phi, RX, ly + 1, ly + 2, ly + 3, lx + 2, ph, gx, gy, lap);
#pragma unroll
        for (int p = 0; p < NS; ++p) { PH[p] = ph[p]; GX[p] = gx[p]; GY[p] = gy[p]; LP[p] = lap[p]; }
        source_terms<NS, MODEL>(P, ph, gx, gy, Rx, Ry);
        mass_flux<NS>(P, gx, gy, Rx, Ry, mx, my);
        s_w[(ly + 1) * BX + lx + 1] = flux_cross(mx, my, upx, upy);
    }
    // w on the one-node ring (u(t-1) of the mirror image, negated across a wall)
    for (int h = t; h < 2 * BX + 2 * PY; h += T) {
        int rx, ry;
        if (h < 2 * BX) {
            const int r = h >= BX;
            rx = h - r * BX - 1;
            ry = r ? He : -1;
        } else {
            const int k = h - 2 * BX;
            ry = k >> 1;
            rx = (k & 1) ? We : -1;
        }
        if (rx >= We + 1 || (h >= 2 * BX && ry >= He)) continue;
        bool fx, fy;
        const int xc = map_axis(x0 + rx, P.nx, P.wall_x, fx), yc = map_axis(y0 + ry, P.ny, P.wall_y, fy);
        const unsigned k = (unsigned)yc * P.nx + xc;
        const float ux = __ldg(P.uin + k), uy = __ldg(P.uin + pl + k), us = fx != fy ? -1.f : 1.f;
        float ph[N], gx[N], gy[N], Qx[NS], Qy[NS], qx, qy;
        window_grad<NS>(s_phi, RX, ry + 1, ry + 2, ry + 3, rx + 2, ph, gx, gy);
        source_terms<NS, MODEL>(P, ph, gx, gy, Qx, Qy);
        mass_flux<NS>(P, gx, gy, Qx, Qy, qx, qy);
        s_w[(ry + 1) * BX + rx + 1] = us * flux_cross(qx, qy, ux, uy);
    }
    __syncthreads();

    // ---------------------------------------------------- stage C
    if (own) {
        float ph[N], gx[N], gy[N], lap[N];
        if constexpr (ST == 0) close_phases<NS>(PH, GX, GY, LP, ph, gx, gy, lap);
        else window_grad_lap<NS>(s_phi, RX, ly + 1, ly + 2, ly + 3, lx + 2, ph, gx, gy, lap);
        const float *w0 = s_w + (ly + 1) * BX + lx + 1;
        const OwnPatch<NS, RX, T> own_node{s_j, s_phi + (ly + 2) * NE * RX, t, lx + 2};
        auto load_g = [&](float (&gv)[9]) {
#pragma unroll
            for (int i = 1; i < 9; ++i) gv[i] = g[i];
        };
        complete_node<NS, ST, TAPE>(P, node, x, y, ph, gx, gy, lap, w0 - BX, w0, w0 + BX, load_g, php, mpx, mpy, Rx,
                                    Ry, mx, my, upx, upy, own_node);
    }
}

template <int NS, int MODEL, int ST, int PX, int PY, int MINB, bool TAPE>
__global__ void __launch_bounds__(PX *PY, MINB) step_patch_kernel(const StepParams P, const int patches_x)
{
    extern __shared__ __align__(16) float smem[];
    pdl_wait();   // launched with launch_pdl
    const int by = blockIdx.x / patches_x, bx = blockIdx.x - by * patches_x;
    step_patch<NS, MODEL, ST, PX, PY, TAPE>(P, bx * PX, by * PY, smem);
}

template <int NS, int MODEL, int ST, int PX, int PY, int MINB, bool TAPE>
cudaError_t launch_patch_variant(const StepParams &p, cudaStream_t st)
{
    constexpr size_t smem = patch_smem_bytes<NS, PX, PY>();
    static_assert(smem <= 48 * 1024, "a patch fits the default shared memory");
    const int bx = (p.nx + PX - 1) / PX, by = (p.ny + PY - 1) / PY;
    return launch_pdl(step_patch_kernel<NS, MODEL, ST, PX, PY, MINB, TAPE>, dim3((unsigned)bx * by), dim3(PX * PY),
                      smem, st, p, bx);
}

// Patch shapes and the blocks per SM they are compiled for.  Narrow patches
// (16 x 8, 128 threads) put a small lattice on more SMs, and one more of
// their blocks fits where registers are short (N = 5, 1024^2: 98.1 us a step
// with four blocks, 91.5 with five).  Wide ones (32 x 8, 256 threads) repeat
// fewer pulls (1.69 against 1.88 per node); they win once they fill the GPU
// where their registers leave three or four blocks (FP32 at N <= 4, and at N =
// 5 with Model A, whose source is lighter; 2048^2 N = 3: 192 against 221 us)
// or where two blocks are all that either shape gets (N = 7, 8: 1024^2 N = 8
// Model A 158 against 168 us).  Patches of 64 x 4, 16 x 16, 32 x 4, 32 x 16,
// 16 x 4 and 8 x 8 nodes were slower than the better of the two by 1 to 60 %.
template <int NS, int MODEL, int ST>
constexpr bool wide_patches()
{
    return NS >= 6 || (ST == 0 ? NS <= 3 || (NS == 4 && MODEL == 0) : NS == 4);
}

template <int NS, int MODEL, int ST, bool TAPE>
cudaError_t launch_patches(const StepParams &p, cudaStream_t st)
{
    constexpr int kNarrowMin = NS <= 3 ? 6 : (NS <= 5 ? 5 : 4), kWideMin = NS <= 2 ? 4 : (NS <= 4 ? 3 : 2);
    constexpr int kFill = 152 * 3 / 2;   // wide patches from 1.5 per SM on (256^2: equal, 300x150: 8 % slower)
    if constexpr (wide_patches<NS, MODEL, ST>()) {
        if ((long long)((p.nx + 31) / 32) * ((p.ny + 7) / 8) >= kFill)
            return launch_patch_variant<NS, MODEL, ST, 32, 8, kWideMin, TAPE>(p, st);
    }
    return launch_patch_variant<NS, MODEL, ST, 16, 8, kNarrowMin, TAPE>(p, st);
}

// Whether an FP32 step runs on patches rather than as a march that updates
// march_nodes nodes (see there): a march spends `gain` of a patch's time on a
// node.  The gain was fitted to both forms of 38 lattices (256 x 1024 to
// 1920^2) per phase count and model; it picks the slower one by 1.3 % at most
// on them (us a step, march / patches, Model B where not said: 256^2 N = 5
// 15.7 / 8.0; 768^2 N = 7 77 / 85, N = 2 24.6 / 21.8; 832^2 N = 8 115 / 123; 1100^2
// N = 5 101 / 108, N = 4 79 / 83; 1024^2 N = 6 Model A 118 / 112; 256 x 4096 N = 5
// 114 / 91; 1472^2 N = 6 222 / 243).  1: patches at every size (2048^2 N = 3 200 /
// 192); so it is for most lattices without row windows (1279^2 N = 6 234 / 203,
// 2045^2 N = 8 761 / 700).
//
// The taping step writes another 8 NS + 12 planes, which patches write best
// where their rows of 32 columns start on a 32-byte sector (nx a multiple of
// 8): there they are ahead at almost any size, elsewhere marches are on large
// lattices (us a step of a taped forward of 8 steps, march / patches, Model B:
// 1024^2 N = 3 86 / 78, N = 5 154 / 127, 1472^2 N = 4 250 / 200; 1100^2 N = 6 189 /
// 223, 868 x 1024 N = 2 53 / 58; 1279^2 N = 3 152 / 164, N = 5 249 / 306, but N = 7
// 408 / 348).
template <int NS, int MODEL, bool TAPE>
inline bool use_patches(const StepParams &p, double march_nodes, bool windows)
{
    if constexpr (TAPE) {
        // nx a multiple of 8; of 4; no row windows
        constexpr bool A = MODEL == 0;
        constexpr double kTape[3][7] = {{1., 1., 1., 1., A ? 1. : .89, 1., A ? .965 : .92},
                                        {.85, .85, 1., A ? 1. : .85, .85, .90, .85},
                                        {.82, .75, .83, .75, .75, 1., 1.}};
        return kTape[windows ? (p.nx % 8 != 0) : 2][NS - 1] * march_nodes >= (double)p.nx * p.ny;
    }
    constexpr double kGain[2][7] = {{.865, 1., .905, .965, .93, .88, .9725}, {.865, 1., .905, .895, .92, .88, .82}};
    const double gain = windows ? kGain[MODEL][NS - 1] : NS == 1 ? .835 : NS == 4 && MODEL == 1 ? .90 : 1.;
    return gain * march_nodes >= (double)p.nx * p.ny;
}

}  // namespace nlbm
