// rt_transport.cu -- one RT step on the GPU (Sec. 2.1 and Sec. 2.2 of the paper).
//
// Packets live in per-particle slots (reception cone b, frequency bin nu), double-buffered
// across hops.  One hop:
//   A  sender side, warp per gas particle (lanes = neighbours): for every packet able to move,
//      the transmission-cone membership of each neighbour (ballot), the equal share w = N/n,
//      and a transposed bitmap (sender, neighbour, nu) -> bins; empty cones request a virtual
//      particle.  Free packets (source packets in the first hop, virtual particles after) do
//      the same with their own neighbour lists and stage their contributions.
//   V  warp per virtual-particle request: position inside the cone (counter-based draws),
//      escape test, exact kNN of the point, SPH-interpolated n_HI, attenuation; absorptions
//      go to the neighbours as fixed-point integer sums (order-independent, so reproducible);
//      the transmitted packet becomes a free packet of the next hop.
//   B  receiver side, a warp per four groups (particle, nu): walks the particles' reverse
//      neighbour lists in sender order, expands the bitmap bits into contributions, attenuates
//      (lane = contribution), picks the reception cone, and merges in a fixed order (sender,
//      slot); then the staged free-packet contributions in (packet, neighbour) order.
//      No floating-point atomics: every sum has one fixed order.
#include <algorithm>
#include <climits>
#include <array>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

#include "rt_knn.cuh"

static const double C_LIGHT = 2.99792458e10;
static const double EV_ERG = 1.602176634e-12;

// the two isotropic direction sets (index 0: 8 directions, 1: 32), FP64 and FP32 copies
__constant__ double c_axd[2][96];
// FP32 copy in global memory for lane-divergent reads, and the candidate table of each set
__device__ float g_axf[2][96];
__device__ unsigned g_bin_tab[2][BIN_TAB_M * BIN_TAB_M];

// Candidate table of a direction set.  Cell (i, j) of the octahedral map covers
// u in [-1 + 2i/M, -1 + 2(i+1)/M], v likewise; its entry lists (one byte each, 0xff unused) the
// directions D_b that can be the nearest for some direction p of the cell, i.e. whose gap
// f_b(p) = p.D_b - max_a p.D_a comes near zero there.  f_b is 2-Lipschitz in p, and the
// inverse map (u, v) -> p is 3-Lipschitz (the point on the octahedron moves by at most
// sqrt(3) |d(u, v)| and has norm >= 1/sqrt(3)), so sampling the cell on a grid of spacing sp
// bounds f_b everywhere in it to within 2 * 3 * sp / sqrt(2) of the sampled maximum.
static void build_bin_table(const double *D, int nax, unsigned *tab) {
    const int M = BIN_TAB_M, S = 17;
    const double sp = 2.0 / (M * (S - 1.0));
    const double thr = -(6.0 * sp / sqrt(2.0) + 1e-3);
    for (int i = 0; i < M; ++i)
        for (int j = 0; j < M; ++j) {
            double fmax[32];
            for (int k = 0; k < nax; ++k) fmax[k] = -1e30;
            for (int a = 0; a < S; ++a)
                for (int b = 0; b < S; ++b) {
                    double u = -1.0 + 2.0 * (i + a / (S - 1.0)) / M;
                    double v = -1.0 + 2.0 * (j + b / (S - 1.0)) / M;
                    double x = u, y = v, z = 1.0 - fabs(u) - fabs(v);
                    if (z < 0.0) {
                        x = (u < 0.0 ? -1.0 : 1.0) * (1.0 - fabs(v));
                        y = (v < 0.0 ? -1.0 : 1.0) * (1.0 - fabs(u));
                    }
                    double nn = sqrt(x * x + y * y + z * z);
                    x /= nn; y /= nn; z /= nn;
                    double sc[32], best = -2.0;
                    for (int k = 0; k < nax; ++k) {
                        sc[k] = x * D[3 * k] + y * D[3 * k + 1] + z * D[3 * k + 2];
                        best = std::max(best, sc[k]);
                    }
                    for (int k = 0; k < nax; ++k) fmax[k] = std::max(fmax[k], sc[k] - best);
                }
            unsigned w = 0xffffffffu;
            int cnt = 0;
            for (int k = 0; k < nax; ++k) {
                if (!(fmax[k] > thr)) continue;
                if (cnt < 4) w = (w & ~(0xffu << (8 * cnt))) | ((unsigned)k << (8 * cnt));
                ++cnt;
            }
            tab[i * M + j] = cnt <= 4 ? w : BIN_TAB_ALL;
        }
}

#define BIN_BAND 2e-5f
// Reception cone of direction d at a particle with rotation R: argmax_b (R^T d) . D_b, first
// maximum on ties.  FP32 scores of the cell's candidates with a guard band on the margin
// between the two best; inside the band (or for a tie) the exact FP64 scan decides.  Every
// direction left out of a cell is more than 1e-3 below the best everywhere in the cell, far
// beyond the FP32 error (~1e-6), so the fast answer is the exact argmax.
template <typename Real>
__device__ inline int bin_fast(const float *Rf, const double *Rd, int ax, int nrc, Real d0,
                               Real d1, Real d2) {
    float f0 = (float)d0, f1 = (float)d1, f2 = (float)d2;
    float e0 = __fmaf_rn(Rf[0], f0, __fmaf_rn(Rf[3], f1, Rf[6] * f2));
    float e1 = __fmaf_rn(Rf[1], f0, __fmaf_rn(Rf[4], f1, Rf[7] * f2));
    float e2 = __fmaf_rn(Rf[2], f0, __fmaf_rn(Rf[5], f1, Rf[8] * f2));
    // octahedral map of e onto [-1, 1]^2
    float is = __fdividef(1.0f, fabsf(e0) + fabsf(e1) + fabsf(e2));
    float u = e0 * is, v = e1 * is;
    if (e2 < 0.0f) {
        float uu = copysignf(1.0f - fabsf(v), u), vv = copysignf(1.0f - fabsf(u), v);
        u = uu;
        v = vv;
    }
    int cu = min(max(__float2int_rd((u + 1.0f) * (0.5f * BIN_TAB_M)), 0), BIN_TAB_M - 1);
    int cv = min(max(__float2int_rd((v + 1.0f) * (0.5f * BIN_TAB_M)), 0), BIN_TAB_M - 1);
    unsigned c = __ldg(&g_bin_tab[ax][cu * BIN_TAB_M + cv]);
    const float *axf = g_axf[ax];
    float b1 = -3.0f, b2 = -3.0f;
    int best = 0;
    int nk = c == BIN_TAB_ALL ? nrc : 4;
#pragma unroll 1
    for (int k = 0; k < nk; ++k) {
        int b = c == BIN_TAB_ALL ? k : (int)((c >> (8 * k)) & 0xffu);
        if (b == 0xff) break;
        float sc = __fmaf_rn(e0, __ldg(&axf[3 * b]),
                             __fmaf_rn(e1, __ldg(&axf[3 * b + 1]), e2 * __ldg(&axf[3 * b + 2])));
        if (sc > b1) { b2 = b1; b1 = sc; best = b; }
        else if (sc > b2) b2 = sc;
    }
    if (b1 - b2 > BIN_BAND) return best;
    return bin_exact(Rd, c_axd[ax], nrc, (double)d0, (double)d1, (double)d2);
}

struct BinTables {
    unsigned t[2][BIN_TAB_M * BIN_TAB_M];
};

void rt_upload_axes() {
    double d[2][96] = {{0}};
    float f[2][96];
    rt_host_axis_set(8, d[0]);
    rt_host_axis_set(32, d[1]);
    for (int a = 0; a < 2; ++a)
        for (int k = 0; k < 96; ++k) f[a][k] = (float)d[a][k];
    static const BinTables *tab = [&d] {   // built once (thread-safe static initialisation)
        BinTables *t = new BinTables;
        build_bin_table(d[0], 8, t->t[0]);
        build_bin_table(d[1], 32, t->t[1]);
        return t;
    }();
    cudaMemcpyToSymbol(c_axd, d, sizeof(d));
    cudaMemcpyToSymbol(g_axf, f, sizeof(f));
    cudaMemcpyToSymbol(g_bin_tab, tab->t, sizeof(tab->t));
}

// Resident 256-thread blocks per SM asked of the hop kernels: four (64 registers a thread)
// for FP32 packets; three for FP64, whose wider values would otherwise spill.  The virtual
// particles take five with FP32 packets (48 registers, some spilled): the extra warps hide
// more latency than the spills cost (measured on the 64^3 step graph).
#define HOP_MINB(Real) (sizeof(Real) == 4 ? 4 : 3)
#ifndef VIRT_MINB_F32
#define VIRT_MINB_F32 5
#endif
#define VIRT_MINB(Real) (sizeof(Real) == 4 ? VIRT_MINB_F32 : 3)
// Largest grids (blocks) of the sender side, the virtual particles and the receiver side.  On
// the sender and receiver sides each block takes a contiguous chunk of the live items; the
// sizes were set by a measured sweep on the 64^3 HII-region step: fewer, longer-lived blocks
// than one per 32 items, while still several blocks per SM turn over during a launch.
#ifndef GRID_A
#define GRID_A (152 * 16)
#endif
#ifndef GRID_V
// one wave with FP32 packets (1.7 with FP64, three blocks an SM: the virtual particles pull from a
// work queue, so the later blocks find what is left)
#define GRID_V (152 * VIRT_MINB_F32)
#endif
#ifndef GRID_B
#define GRID_B (152 * 8)
#endif
#define GRID_F (152 * 4)   // free-packet senders: one wave (1.3 with FP64)

template <typename Real> struct Slots {
    Real *N, *X, *Y, *Z, *C, *E;
    __device__ __forceinline__ Slots(const DevPtrs &P, int b) {
        N = (Real *)P.sl[b][0]; X = (Real *)P.sl[b][1]; Y = (Real *)P.sl[b][2];
        Z = (Real *)P.sl[b][3]; C = (Real *)P.sl[b][4]; E = (Real *)P.sl[b][5];
    }
};

// phase-A record of a slot: (w, d, clock, eps) in one aligned piece of 8 Real, and with `sg`
// (a slot of a shared frequency bin) the packet's mean cross-section in the seventh
__device__ __forceinline__ void rec_store(void *rec, long long s, float w, float d0, float d1,
                                          float d2, float c, float e, bool sg, float sig) {
    float4 *p = (float4 *)rec + 2 * s;
    p[0] = make_float4(w, d0, d1, d2);
    if (sg) p[1] = make_float4(c, e, sig, 0.0f);
    else *(float2 *)(p + 1) = make_float2(c, e);
}
__device__ __forceinline__ void rec_store(void *rec, long long s, double w, double d0, double d1,
                                          double d2, double c, double e, bool sg, double sig) {
    double2 *p = (double2 *)rec + 4 * s;
    p[0] = make_double2(w, d0);
    p[1] = make_double2(d1, d2);
    p[2] = make_double2(c, e);
    if (sg) p[3] = make_double2(sig, 0.0);
}
__device__ __forceinline__ void rec_load(const void *rec, long long s, float &w, float &d0,
                                         float &d1, float &d2, float &c, float &e, bool sg,
                                         float &sig) {
    const float4 *p = (const float4 *)rec + 2 * s;
    float4 a = p[0];
    w = a.x; d0 = a.y; d1 = a.z; d2 = a.w;
    if (sg) {
        float4 b = p[1];
        c = b.x; e = b.y; sig = b.z;
    } else {
        float2 b = *(const float2 *)(p + 1);
        c = b.x; e = b.y;
    }
}
__device__ __forceinline__ void rec_load(const void *rec, long long s, double &w, double &d0,
                                         double &d1, double &d2, double &c, double &e, bool sg,
                                         double &sig) {
    const double2 *p = (const double2 *)rec + 4 * s;
    double2 a = p[0], b = p[1], d = p[2];
    w = a.x; d0 = a.y; d1 = b.x; d2 = b.y; c = d.x; e = d.y;
    if (sg) sig = p[3].x;
}

// Quotients with a shared divisor, correctly rounded like a division each (div_by_rcp): an FP64
// division takes about ten FP64 instructions, a further quotient by the same divisor three.  The
// plain division where an operand is so large or small that the exact remainder could leave
// the range.  (A zero numerator of either sign gives +0; every sum that takes it starts at +0.)
__device__ __forceinline__ bool in_range(double a) {   // 2^-400 <= |a| < 2^401
    return (((unsigned)__double2hiint(a) >> 20) & 0x7ffu) - 623u < 801u;
}
__device__ __forceinline__ double quot(double a, double b, double y) {   // y = 1 / b, rounded
    bool zero = (__double_as_longlong(a) << 1) == 0ll;
    return (in_range(a) || zero) && in_range(b) ? div_by_rcp(a, b, y) : a / b;
}

// unit direction of a packet from its summed momentum M (the luminosity-weighted mean
// direction of merged packets, Sec. 2.1, Fig. 1b)
__device__ __forceinline__ void packet_dir(double Mx, double My, double Mz, double &d0, double &d1,
                                           double &d2) {
    double nn = sqrt(Mx * Mx + My * My + Mz * Mz);
    if (nn > 0.0) {
        double y = __drcp_rn(nn);
        d0 = quot(Mx, nn, y); d1 = quot(My, nn, y); d2 = quot(Mz, nn, y);
    } else {
        d0 = 1.0; d1 = 0.0; d2 = 0.0;
    }
}

// FP32: normalised photon counts can be small enough for |M|^2 to underflow, so scale first.
// Every operation is a correctly rounded IEEE single-precision operation in a fixed order
// (reciprocal, products, (a^2 + b^2) + c^2, square root, reciprocal, products), so the FP32
// direction is a reproducible function of the stored momentum: the exact cone test (FP64, on
// this direction) then decides every membership the same way wherever it is evaluated.
__device__ __forceinline__ void packet_dir(float Mx, float My, float Mz, float &d0, float &d1,
                                           float &d2) {
    float s = fmaxf(fabsf(Mx), fmaxf(fabsf(My), fabsf(Mz)));
    if (s > 0.0f) {
        float is = __frcp_rn(s);
        float a = __fmul_rn(Mx, is), b = __fmul_rn(My, is), c = __fmul_rn(Mz, is);
        float q = __fadd_rn(__fadd_rn(__fmul_rn(a, a), __fmul_rn(b, b)), __fmul_rn(c, c));
        float rn = __frcp_rn(__fsqrt_rn(q));
        d0 = __fmul_rn(a, rn); d1 = __fmul_rn(b, rn); d2 = __fmul_rn(c, rn);
    } else {
        d0 = 1.0f; d1 = 0.0f; d2 = 0.0f;
    }
}

// a / b: IEEE division on the FP64 path (the oracle's arithmetic), a times the correctly
// rounded reciprocal on the FP32 path
template <typename Real> __device__ __forceinline__ Real rdiv(Real a, Real b);
template <> __device__ __forceinline__ double rdiv<double>(double a, double b) { return a / b; }
template <> __device__ __forceinline__ float rdiv<float>(float a, float b) { return a * __frcp_rn(b); }

// mean clock and energy of a packet: C / N and E / N (rdiv's arithmetic)
__device__ __forceinline__ void means(double C, double E, double N, double &c, double &e) {
    double y = __drcp_rn(N);
    c = quot(C, N, y);
    e = quot(E, N, y);
}
__device__ __forceinline__ void means(float C, float E, float N, float &c, float &e) {
    float y = __frcp_rn(N);
    c = C * y;
    e = E * y;
}
// the same as IEEE quotients in both precisions
__device__ __forceinline__ void ratios(double C, double E, double N, double &c, double &e) {
    means(C, E, N, c, e);
}
__device__ __forceinline__ void ratios(float C, float E, float N, float &c, float &e) {
    c = C / N;
    e = E / N;
}
// l / c: the time a packet takes for the length l
__device__ __forceinline__ double light_time(double l) { return quot(l, C_LIGHT, 1.0 / C_LIGHT); }
__device__ __forceinline__ float light_time(float l) {
    const float c = (float)C_LIGHT, y = 1.0f / c;
    if (!(fabsf(l) > 1e-15f)) return l / c;
    float q = __fmul_rn(l, y);
    return __fmaf_rn(__fmaf_rn(-q, c, l), y, q);
}

// precision-matched constants: FP64 values on the FP64 path, FP32 copies on the FP32 path
template <typename Real> __device__ __forceinline__ Real box_unit(const DevPtrs &P, int b);
template <> __device__ __forceinline__ double box_unit<double>(const DevPtrs &P, int b) { return P.box_u[b]; }
template <> __device__ __forceinline__ float box_unit<float>(const DevPtrs &P, int b) { return P.box_uf[b]; }
template <typename Real> __device__ __forceinline__ Real sigma_of(const DevPtrs &P, int nu);
template <> __device__ __forceinline__ double sigma_of<double>(const DevPtrs &P, int nu) { return P.sigma[nu]; }
template <> __device__ __forceinline__ float sigma_of<float>(const DevPtrs &P, int nu) { return P.sigmaf[nu]; }
// the cross-section of a bin in the unit of the shared-bin fields (sunit)
template <typename Real> __device__ __forceinline__ Real sigma_units(const DevPtrs &P, int nu);
template <> __device__ __forceinline__ double sigma_units<double>(const DevPtrs &P, int nu) {
    return P.sigma[nu] / P.sunit;
}
template <> __device__ __forceinline__ float sigma_units<float>(const DevPtrs &P, int nu) {
    return (float)(P.sigma[nu] / P.sunit);
}
template <typename Real> __device__ __forceinline__ Real to_real(long long v);
template <> __device__ __forceinline__ double to_real<double>(long long v) { return (double)v; }
template <> __device__ __forceinline__ float to_real<float>(long long v) { return i64_to_f(v); }

__device__ __forceinline__ unsigned long long to_fixed(double v) { return (unsigned long long)llrint(v); }
__device__ __forceinline__ unsigned long long to_fixed(float v) { return f2u64_rz(v + 0.5f); }

// escaped photons in the fixed-point unit of the box's escape tally
__device__ __forceinline__ unsigned long long esc_fixed(double N, const DevPtrs &P, int box) {
    return (unsigned long long)llrint(N * P.norm[box] / P.ref[box] * FX_ESC_SCALE);
}
__device__ __forceinline__ unsigned long long esc_fixed(float N, const DevPtrs &P, int box) {
    return f2u64_rz(N * P.escf[box] + 0.5f);
}

// ------------------------------------------------------------------------------------------
// per-step kernels
// ------------------------------------------------------------------------------------------
__global__ void k_rotate(DevPtrs P) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long step = P.cnt[CNT_STEP];
    long long nsrc = (long long)P.ns * P.K;
    if (i < P.n) {
        double R[9];
        random_rotation(P.seed, 1u, (unsigned)step, (unsigned)(step >> 32),
                        (unsigned)gid_of(P, i, P.pbox[i]), R);
#pragma unroll
        for (int a = 0; a < 9; ++a) { P.R[i * 9 + a] = R[a]; P.Rf[i * 9 + a] = (float)R[a]; }
    } else if (i < P.n + nsrc) {
        long long t = i - P.n;
        int j = (int)((unsigned)t / (unsigned)P.K), k = (int)((unsigned)t % (unsigned)P.K);
        double R[9];
        random_rotation(P.seed, 2u, (unsigned)step, (unsigned)k, (unsigned)P.sid[j], R);
#pragma unroll
        for (int a = 0; a < 9; ++a) P.Rs[t * 9 + a] = R[a];
    }
}

// Start of step: clock reset and re-binning of held packets into the new reception cones.
template <typename Real, int NRC>
__global__ void k_rebin(DevPtrs P) {
    long long key = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (key >= P.n * P.nf) return;
    int cur = (int)P.cnt[CNT_CUR];
    unsigned o = P.occ[cur][key];
    if (!o) { P.act[cur][key] = 0; return; }
    long long i = (unsigned)key / (unsigned)P.nf;   // keys < 2^31: 32-bit division
    int nu = (int)((unsigned)key % (unsigned)P.nf);
    Slots<Real> S(P, cur);
    long long s0 = i * P.S + (long long)nu * NRC;
    Real nN[NRC], nX[NRC], nY[NRC], nZ[NRC], nE[NRC], nG[NRC];
    Real oN[NRC], oX[NRC], oY[NRC], oZ[NRC], oE[NRC], oG[NRC];
    // a shared frequency bin carries the cross-section sums of bin 0 along
    Real *SG = (P.shared && nu == 0) ? (Real *)P.slG[cur] + i * NRC : nullptr;
    for (int b = 0; b < NRC; ++b) {
        nN[b] = nX[b] = nY[b] = nZ[b] = nE[b] = nG[b] = Real(0);
        if ((o >> b) & 1) {
            oN[b] = S.N[s0 + b]; oX[b] = S.X[s0 + b]; oY[b] = S.Y[s0 + b];
            oZ[b] = S.Z[s0 + b]; oE[b] = S.E[s0 + b];
            oG[b] = SG ? SG[b] : Real(0);
        }
    }
    const double *Rd = P.R + i * 9;
    const float *Rf = P.Rf + i * 9;
    for (int b = 0; b < NRC; ++b) {
        if (!((o >> b) & 1) || !(oN[b] > Real(0))) continue;
        Real d0, d1, d2;
        packet_dir(oX[b], oY[b], oZ[b], d0, d1, d2);
        int nb = bin_fast<Real>(Rf, Rd, P.ax_rc, NRC, d0, d1, d2);
        nN[nb] += oN[b]; nX[nb] += oX[b]; nY[nb] += oY[b]; nZ[nb] += oZ[b]; nE[nb] += oE[b];
        nG[nb] += oG[b];
    }
    unsigned no = 0;
    for (int b = 0; b < NRC; ++b) {
        if (nN[b] > Real(0)) {
            no |= 1u << b;
            S.N[s0 + b] = nN[b]; S.X[s0 + b] = nX[b]; S.Y[s0 + b] = nY[b];
            S.Z[s0 + b] = nZ[b]; S.C[s0 + b] = Real(0); S.E[s0 + b] = nE[b];
            if (SG) SG[b] = nG[b];
        }
    }
    P.occ[cur][key] = no;
    P.act[cur][key] = no;   // clocks restart: every held packet can move again
}

// the direction of a set opposite to direction b (both sets are symmetric about the origin)
__device__ __forceinline__ int axis_opposite(int nax, int b) {
    if (nax == 8) return 7 - b;
    if (b >= 12 && b < 20) return 31 - b;   // the cube diagonals of the 32: 12 + (7 - (b - 12))
    return b ^ 3;                           // vertex groups of four: both signs flip
}

// The step's deposit words back to zero: key by key across the grid (coalesced), and only those
// the packet precision uses.  A kernel of its own: in the step graph it runs beside the rotations,
// which the FP64 pipe bounds, and takes their memory time (2.1 M particles with hardly any packets:
// the step 0.6% shorter).
template <typename Real>
__global__ void k_clear_deposits(DevPtrs P) {
    for (long long key = (long long)blockIdx.x * blockDim.x + threadIdx.x; key < P.n * P.nf;
         key += (long long)gridDim.x * blockDim.x) {
        if (sizeof(Real) == 8) {
            P.abs[key] = 0.0; P.absE[key] = 0.0; P.pass[key] = 0.0;
        } else {
            P.passf[key] = 0.0f;
        }
        P.fx_abs[key] = 0ull; P.fx_lo[key] = 0ull; P.fx_E[key] = 0ull;
    }
}

// Recombination emission into the reception cones, frozen n_HI.  Bound by FP64 (16 cycles of an
// SM per warp instruction): the rotated axes are computed for one of each opposite pair, and
// the particles' volumes, which a step does not change, come from the upload.  The 64^3 HII
// region, 32 cones, with the deposit words cleared: 420 us with an axis a cone and strided
// clearing, 203 us in one kernel.
template <typename Real, int NRC>
__global__ void k_emit_rec(DevPtrs P, int *lens, int np) {
    long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) {   // the hop loop starts with the step's np emitted packets in free buffer 0
        lens[0] = np;
        P.cnt[CNT_FCUR] = 0;
    }
    if (i >= P.n) return;
    int cur = (int)P.cnt[CNT_CUR];
    double nm = P.norm[P.pbox[i]];
    double x = P.xHI[i], nH = P.nH[i], NH = P.NH[i];
    double nHI = __dmul_rn(x, nH);
    P.nHI[i] = nHI;
    double NHI = x * NH;
    ((Real *)P.nHIr)[i] = (Real)nHI;
    pv<Real>(P, i, PV_NHI) = (Real)nHI;
    pv<Real>(P, i, PV_DEP) = NHI > 0.0 ? (Real)(FX_ABS_SCALE * nm / NHI) : Real(0);
    pv<Real>(P, i, PV_DEPE) = NHI > 0.0 ? (Real)(FX_E_SCALE * nm * P.eunit / (NHI * EV_ERG)) : Real(0);
    double Nr = P.Nrec[i];
    if (!(Nr > 0.0) || P.rec_mode == RT_REC_EMISSION_CONES) return;
    double e_phys = Nr / (double)NRC;
    Real e = (Real)(e_phys / nm);
    Real epsr = (Real)(P.epsrec[i] / P.eunit);
    int nu = P.rbin;       // the recombination bin, or source bin 0 when the bin is shared
    long long key = i * P.nf + nu;
    unsigned o = P.occ[cur][key], a = P.act[cur][key];
    Slots<Real> S(P, cur);
    long long s0 = i * P.S + (long long)nu * NRC;
    // shared bin: each cone gains e sigma_rec of cross-section sum
    Real *SG = P.shared ? (Real *)P.slG[cur] + i * NRC : nullptr;
    Real eg = e * (Real)(P.sigma_rec / P.sunit);
    double R[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) R[k] = P.R[i * 9 + k];
    auto emit = [&](int bb, Real A0, Real A1, Real A2) {
        long long s = s0 + bb;
        if ((o >> bb) & 1) {
            S.N[s] += e; S.X[s] += e * A0; S.Y[s] += e * A1;
            S.Z[s] += e * A2; S.E[s] += e * epsr;
            if (SG) SG[bb] += eg;
        } else {
            S.N[s] = e; S.X[s] = e * A0; S.Y[s] = e * A1;
            S.Z[s] = e * A2; S.C[s] = Real(0); S.E[s] = e * epsr;
            if (SG) SG[bb] = eg;
        }
    };
    for (int bb = 0; bb < NRC; ++bb) {
        int ob = axis_opposite(NRC, bb);
        if (ob < bb) continue;
        double A[3];
        rot_apply(R, c_axd[P.ax_rc] + 3 * bb, A);
        Real A0 = (Real)A[0], A1 = (Real)A[1], A2 = (Real)A[2];
        emit(bb, A0, A1, A2);
        emit(ob, -A0, -A1, -A2);
    }
    if (e > Real(0)) {
        const unsigned all = NRC == 32 ? FULLMASK : (1u << (NRC & 31)) - 1u;
        o |= all;
        a |= all;
    }
    P.occ[cur][key] = o;
    P.act[cur][key] = a;
}

// Source packets of the step: K emissions x n_freq_src bins x n_ec cones per source, written
// to free buffer 0 (the first hop's).
template <typename Real>
__global__ void k_emit_src(DevPtrs P) {
    long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long per_src = (long long)P.K * P.nfs * P.nec;
    if (p >= (long long)P.ns * per_src) return;
    unsigned ps = (unsigned)per_src, tt = (unsigned)(p % ps);
    int j = (int)((unsigned)p / ps);
    int k = (int)(tt / (unsigned)(P.nfs * P.nec));
    int nu = (int)((tt / (unsigned)P.nec) % (unsigned)P.nfs);
    int e = (int)(tt % (unsigned)P.nec);
    FreeBuf F = P.fr[0];
    int b = P.sbox[j];
    // a gated source emits only while its nearest gas particle is more than half ionised; a
    // directed source sends one packet per emission and frequency (cone 0) along its direction
    const double *dir = P.sdir + 3 * (long long)j;
    bool directed = dir[0] != 0.0 || dir[1] != 0.0 || dir[2] != 0.0;
    bool on = !P.sgate[j] || P.xHI[P.snbr[(long long)j * P.kn]] < 0.5;
    double nd = P.ndot[(long long)j * P.nfs + nu];
    double N = 0.0, d[3];
    if (directed) {
        if (on && e == 0) N = __dmul_rn(nd, P.dt_em);
        d[0] = dir[0]; d[1] = dir[1]; d[2] = dir[2];
    } else {
        if (on) N = __ddiv_rn(__dmul_rn(nd, P.dt_em), (double)P.nec);
        rot_apply(P.Rs + ((long long)j * P.K + k) * 9, c_axd[P.ax_ec] + 3 * e, d);
    }
    F.box[p] = b;
    F.qx[p] = P.sqx[j]; F.qy[p] = P.sqy[j]; F.qz[p] = P.sqz[j];
    for (int a = 0; a < P.kn; ++a) F.nbr[p * P.kn + a] = P.snbr[(long long)j * P.kn + a];
    F.h2[p] = P.sh2[j];
    ((Real *)F.N)[p] = (Real)(N / P.norm[b]);
    ((Real *)F.dx)[p] = (Real)d[0];
    ((Real *)F.dy)[p] = (Real)d[1];
    ((Real *)F.dz)[p] = (Real)d[2];
    ((Real *)F.clock)[p] = Real(0);
    ((Real *)F.eps)[p] = (Real)(P.eps[nu] / P.eunit);
    if (P.shared) ((Real *)F.sig)[p] = sigma_units<Real>(P, nu);
    F.nu[p] = nu;
    // identity (source, emission, frequency, cone), with the source's identity
    F.okey[p] = RT_OKEY_GEN | (unsigned long long)p;
    F.fid[p] = (1ull << 62) |
               ((((unsigned long long)P.sid[j] * P.K + k) * P.nfs + nu) * P.nec + e);
}

// The original implementation of recombination radiation (Sec. 2.2): particle i emits, K
// times a step, n_ec packets of N_rec / (K n_ec) photons along its emission axes, rotated at
// random before each emission; they are free packets at the particle's position with its
// neighbour list, written to free buffer 0 after the source packets (index
// base + (i K + k) n_ec + e).
// Particles without recombination photons leave packets of N = 0, which never move.
template <typename Real>
__global__ void k_emit_rec_cones(DevPtrs P, long long base) {
    long long p = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    long long per = (long long)P.K * P.nec;
    if (p >= P.n * per) return;
    long long step = P.cnt[CNT_STEP];
    long long i = p / per;
    int k = (int)((p % per) / P.nec), e = (int)(p % P.nec);
    FreeBuf F = P.fr[0];
    long long f = base + p;
    const int4 q = P.q4[i];
    const int b = q.w;
    double Nr = P.Nrec[i];
    double N = Nr > 0.0 ? __ddiv_rn(Nr, (double)per) : 0.0;
    double R[9], d[3];
    const unsigned long long gi = gid_of(P, i, b);
    random_rotation(P.seed, 4u, (unsigned)step, (unsigned)k, (unsigned)gi, R);
    rot_apply(R, c_axd[P.ax_ec] + 3 * e, d);
    F.box[f] = b;
    F.qx[f] = q.x; F.qy[f] = q.y; F.qz[f] = q.z;
    for (int a = 0; a < P.kn; ++a) F.nbr[f * P.kn + a] = P.nbr[i * P.kn + a];
    F.h2[f] = P.h2[i];
    ((Real *)F.N)[f] = (Real)(N / P.norm[b]);
    ((Real *)F.dx)[f] = (Real)d[0];
    ((Real *)F.dy)[f] = (Real)d[1];
    ((Real *)F.dz)[f] = (Real)d[2];
    ((Real *)F.clock)[f] = Real(0);
    ((Real *)F.eps)[f] = (Real)(P.epsrec[i] / P.eunit);
    if (P.shared) ((Real *)F.sig)[f] = (Real)(P.sigma_rec / P.sunit);
    F.nu[f] = P.rbin;
    F.okey[f] = RT_OKEY_GEN | (unsigned long long)f;
    F.fid[f] = (2ull << 62) | ((gi * P.K + k) * P.nec + e);   // (particle, emission, cone)
}

// ------------------------------------------------------------------------------------------
// hop kernels
// ------------------------------------------------------------------------------------------
// inclusive prefix sum over the lanes (of packed fields that do not overflow)
__device__ __forceinline__ unsigned lane_scan(unsigned v) {
    int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        unsigned t = __shfl_up_sync(FULLMASK, v, o);
        if (lane >= o) v += t;
    }
    return v;
}

// The packet of a slot as the sender side reads it: photon count, direction, mean clock and
// energy, and in a shared frequency bin the mean cross-section.
template <typename Real> struct SentPacket {
    Real N, d0, d1, d2, C, E, sg;
};

// Sender side.  A warp takes a few consecutive particles at a time (`per`, at most 32 / n_freq),
// lane = (particle, frequency) word of packets able to move; their packets are taken 32 at a
// time (lane = packet: load, direction, clock), then tested one after the other against the
// neighbours of their particle (lane = neighbour k: cone membership, ballot).  For each
// (frequency, neighbour) the bits of the packets whose cone holds the neighbour go to the
// neighbour's receiver-ordered bitmap word; empty cones become virtual-particle requests, in no
// particular order: what depends on an order of the packets they become orders itself (FreeBuf
// okey).
// What bounds it: the latency of the dependent gathers and instruction issue; a particle holds
// few packets able to move (2.5 with 8 cones behind a fast front, 3.8 over 9 frequencies in the
// HII region), so with a particle of its own most lanes of a warp idled in the packet part
// (FP64 there: 16 cycles of an SM an instruction).  The next particle's neighbours are loaded
// while the current one's packets are tested; what a test needs of a neighbour alone (inverse
// distance) is computed once a particle.  Measured per step against a warp a particle: 2.1 M
// particles behind a fast front, 8 cones, 139 -> 78 ms; 64^3 HII region, 32 cones, 13.1 -> 10.7 ms;
// the FP64 path at 32^3 8.3 -> 5.8 ms; a 64^3 box with hardly any packets 1.77 -> 0.92 ms.
// cur: the slot buffer holding the hop's packets.  Receivers of a bitmap word are flagged in
// `touched` (cleared again by the work-list kernel).
// SH: the shared frequency bin (a separate instance keeps its code out of the common case)
// WIDE: more than 32 frequencies, in several launches a hop (an instance of its own likewise): one
// serves the frequencies nu0 .. nu0 + nfl - 1 (at most 32, a lane a word).  Each bitmap word belongs
// to one frequency, so it is still written once.
// lens: the hop's counts (the request list is lens[2] long); null: no requests (inspection)
template <typename Real, int NRC, bool SH, bool WIDE>
__global__ void __launch_bounds__(256, HOP_MINB(Real)) k_phaseA(DevPtrs P, int cur, int per, int nu0w,
                                                                int nflw, int *lens) {
    const int nu0 = WIDE ? nu0w : 0, nfl = WIDE ? nflw : P.nf;
    __shared__ unsigned slist[8][32];
    __shared__ unsigned sreq[8][64];   // requests not yet in the list
    __shared__ int snext, scnt[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned *list = slist[wid], *rq = sreq[wid];
    int nrq = 0;
    const float cf = 1.0f - 2.0f / (float)P.ntc;
    const long long nrev = P.n * P.kn;
    const unsigned pmask = nfl < 32 ? (1u << nfl) - 1u : FULLMASK;   // a particle's words
    long long ncon = 0;
    int nsend = 0;
    // each block takes one contiguous chunk of particles; its warps pull from it through a
    // shared counter, so that they finish together (particles hold from none to hundreds of
    // packets)
    long long chunk = (P.n + gridDim.x - 1) / gridDim.x;
    const long long ib0 = (long long)blockIdx.x * chunk;
    const long long ib1 = ib0 + chunk < P.n ? ib0 + chunk : P.n;
    if (threadIdx.x == 0) snext = 0;
    __syncthreads();
    const int lp = lane / nfl, lnu = nu0 + lane - lp * nfl;  // the lane's particle and frequency
    auto words = [&](long long i) {
        return (i + lp < ib1 && lp < per) ? P.act[cur][(i + lp) * P.nf + lnu] : 0u;
    };
    // turns a warp takes at once: up to four, whose words it loads together (where nothing moves it
    // goes on after one load), fewer towards the end of the chunk, so that the warps end together
    auto at_once = [&](long long left) { return (int)max(1ll, min(4ll, left / (16 * per))); };
    int turns = at_once(chunk);
    for (;;) {
        long long i0 = 0;
        if (lane == 0) i0 = ib0 + atomicAdd(&snext, per * turns);
        i0 = __shfl_sync(FULLMASK, i0, 0);
        if (i0 >= ib1) break;
        const int now = turns;
        turns = at_once(ib1 - i0);
        unsigned w4[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) w4[u] = u < now ? words(i0 + u * per) : 0u;
        if (__ballot_sync(FULLMASK, (w4[0] | w4[1] | w4[2] | w4[3]) != 0u) == 0u) continue;
#pragma unroll 1
        for (int u = 0; u < now; ++u) {
        const unsigned aw = u < 2 ? (u == 0 ? w4[0] : w4[1]) : (u == 2 ? w4[2] : w4[3]);
        const long long ic = i0 + u * per;
        const unsigned moving = __ballot_sync(FULLMASK, aw != 0u);
        if (moving == 0u) continue;
        bool sends = lane < per && ((moving >> (lane * nfl)) & pmask) != 0u;
        if (WIDE)                             // a particle counts once, in its first launch
            for (int nu = 0; nu < nu0; ++nu)
                sends = sends && P.act[cur][(ic + lane) * P.nf + nu] == 0u;
        nsend += sends;
        const unsigned cnt = (unsigned)__popc(aw);
        const unsigned incl = lane_scan(cnt);
        const int total = (int)__shfl_sync(FULLMASK, incl, 31);
        // the current particle's neighbour of this lane, and the next one's
        float ex = 0.f, ey = 0.f, ez = 0.f;   // offset, place in the reverse lists, index
        int rp = 0, nb = 0, nbn = 0;
        float4 edn = make_float4(0.f, 0.f, 0.f, 0.f);
        float ir = 0.f;
        bool valid = false;
        int curp = -1;                    // the current particle (of the turn's)
        unsigned word = 0u;               // the bitmap word under construction
        int wnu = -1;                     // and its frequency
        auto fetch = [&](int p) {
            if (lane < P.kn) {
                long long f = (ic + p) * P.kn + lane;
                edn = __ldg(P.fwd4 + f);
                nbn = __ldg(P.nbr + f);
            }
        };
        auto flush = [&]() {
            if (word) {
                P.bm[(long long)wnu * nrev + rp] = word;
                P.touched[(long long)nb * P.nf + wnu] = 1;
            }
            word = 0u;
        };
        for (int cb = 0; cb < total; cb += 32) {
            int p = (int)(incl - cnt) - cb;
            for (unsigned x = aw; x; x &= x - 1u, ++p)
                if (p >= 0 && p < 32) list[p] = (unsigned)(__ffs(x) - 1) | (unsigned)lane << 5;
            __syncwarp();
            const int nk = min(32, total - cb);
            const bool has = lane < nk;
            const unsigned code = list[has ? lane : 0];
            const int row = (int)(code >> 5), ob = (int)(code & 31u);
            const int op = __shfl_sync(FULLMASK, lp, row), onu = __shfl_sync(FULLMASK, lnu, row);
            __syncwarp();
            // the runs of packets of one particle
            const int prevp = __shfl_up_sync(FULLMASK, op, 1);
            unsigned first = __ballot_sync(FULLMASK, has && (lane == 0 ? op != curp : op != prevp));
            if (first) fetch(__shfl_sync(FULLMASK, op, __ffs(first) - 1));
            const long long s = (ic + op) * P.S + (long long)onu * NRC + ob;
            SentPacket<Real> K = {Real(0), Real(1), Real(0), Real(0), Real(0), Real(0), Real(0)};
            const bool sgs = SH && onu == 0;   // a slot of the shared bin: its mean cross-section
            if (has) {
                Slots<Real> S(P, cur);
                K.N = S.N[s];
                packet_dir(S.X[s], S.Y[s], S.Z[s], K.d0, K.d1, K.d2);
                K.C = S.C[s];
                K.E = S.E[s];
                if (sgs) K.sg = ((Real *)P.slG[cur])[(ic + op) * NRC + ob] / K.N;
            }
            const float f0 = (float)K.d0, f1 = (float)K.d1, f2 = (float)K.d2;
            int my_cm = 0;
            // the packets one after the other (lane = neighbour k): cone membership; the bitmap
            // word of lane k collects, frequency by frequency, the bins whose cone holds k (a
            // word continues across turns of 32 packets while its particle and frequency do)
            for (int t = 0; t < nk; ++t) {
                if ((first >> t) & 1u) {
                    flush();
                    ex = edn.x; ey = edn.y; ez = edn.z;
                    rp = __float_as_int(edn.w);
                    nb = nbn;
                    curp = __shfl_sync(FULLMASK, op, t);
                    wnu = -1;
                    valid = lane < P.kn && (ex != 0.f || ey != 0.f || ez != 0.f);
                    ir = rsqrtf(__fmaf_rn(ex, ex, __fmaf_rn(ey, ey, ez * ez)));
                    unsigned later = first & (0xfffffffeu << t);
                    if (later) fetch(__shfl_sync(FULLMASK, op, __ffs(later) - 1));
                }
                const float e0 = __shfl_sync(FULLMASK, f0, t), e1 = __shfl_sync(FULLMASK, f1, t),
                            e2 = __shfl_sync(FULLMASK, f2, t);
                const int unu = __shfl_sync(FULLMASK, onu, t), ub = __shfl_sync(FULLMASK, ob, t);
                const float cs = __fmaf_rn(ex, e0, __fmaf_rn(ey, e1, ez * e2)) * ir;
                bool in = valid && cs > cf + CONE_BAND;
                const bool amb = valid && !in && !(cs < cf - CONE_BAND);
                if (__any_sync(FULLMASK, amb)) {   // inside the guard band: the exact test
                    const Real x0 = __shfl_sync(FULLMASK, K.d0, t), x1 = __shfl_sync(FULLMASK, K.d1, t),
                               x2 = __shfl_sync(FULLMASK, K.d2, t);
                    if (amb)
                        in = cone_exact((int)ex, (int)ey, (int)ez, (double)x0, (double)x1,
                                        (double)x2, P.ntc);
                }
                const unsigned m = __ballot_sync(FULLMASK, in);
                if (lane == t) my_cm = __popc(m);
                if (unu != wnu) {
                    flush();
                    wnu = unu;
                }
                if (in) word |= 1u << ub;
            }
            ncon += my_cm;
            if (has) {
                if (my_cm > 0) {
                    Real c, e;
                    means(K.C, K.E, K.N, c, e);
                    rec_store(P.rec, s, rdiv<Real>(K.N, (Real)my_cm), K.d0, K.d1, K.d2, c, e, sgs, K.sg);
                }
            }
            // packets without a member request a virtual particle
            const unsigned rm = lens ? __ballot_sync(FULLMASK, has && my_cm == 0) : 0u;
            if (rm) {
                if ((rm >> lane) & 1u) rq[nrq + __popc(rm & ((1u << lane) - 1u))] = (unsigned)s;
                nrq += __popc(rm);
                __syncwarp();
                if (nrq >= 32) {
                    int base = 0;
                    if (lane == 0) base = atomicAdd(&lens[2], 32);
                    base = __shfl_sync(FULLMASK, base, 0);
                    const unsigned v0 = rq[lane], v1 = rq[32 + lane];
                    if (base + lane < P.F_cap) P.req[base + lane] = v0;
                    __syncwarp();
                    nrq -= 32;
                    if (lane < nrq) rq[lane] = v1;
                    __syncwarp();
                }
            }
        }
        // every word starts the hop at zero (the receiver side clears the words it reads), and
        // each (frequency, neighbour) word is written once: a plain store
        flush();
        }
    }
    if (lens) {   // what is left of the block's requests, in one piece
        if (lane == 0) scnt[wid] = nrq;
        __syncthreads();
        int before = 0, all = 0;
        for (int k = 0; k < 8; ++k) {
            if (k < wid) before += scnt[k];
            all += scnt[k];
        }
        __syncthreads();
        if (threadIdx.x == 0 && all) snext = atomicAdd(&lens[2], all);
        __syncthreads();
        if (lane < nrq && snext + before + lane < P.F_cap) P.req[snext + before + lane] = rq[lane];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ncon += __shfl_down_sync(FULLMASK, ncon, o);
    nsend = __reduce_add_sync(FULLMASK, nsend);
    if (lane == 0 && ncon) atomicAdd((unsigned long long *)&P.cnt[CNT_GCON], (unsigned long long)ncon);
    // the senders of a hop are the previous hop's receivers of packets able to move
    if (lane == 0 && nsend && cnt_word(P, CNT_HOP) != 0u)
        atomicAdd((unsigned long long *)&P.cnt[CNT_ACTP], (unsigned long long)nsend);
}

// Free packets (source packets in the first hop, virtual particles after): a warp takes up to 32
// at a time (lane = packet), tests them one after the other against their own neighbour lists
// (lane = neighbour; the next packets' neighbours and their positions are loaded ahead), and
// collects the members of their cones in a list.  32 members at a time (lane = member) become
// staged contributions, at a position from one counter: a packet has about one member, so a
// warp of its own computed one contribution with one lane.  The position is arbitrary; a
// contribution names its packet (st_pkt), by whose order the receiver orders its segment, and its
// place among the receiver's (st_rank, the count before it).  A packet without a member
// requests a virtual particle.  Measured per step against two kernels and a prefix sum with a
// warp a packet: 64^3 HII region 7.4 -> 3.6 ms, the FP64 path at 32^3 4.7 -> 1.8 ms.
template <typename Real, int NRC, bool BAR, bool SH>
__global__ void __launch_bounds__(256, HOP_MINB(Real)) k_free(DevPtrs P, int fcur, int *lens) {
    __shared__ unsigned smj[8][64];   // member: particle, and the packet's member count - 1 above bit 27
    __shared__ int smf[8][64];        // its packet
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    unsigned *mj = smj[wid];
    int *mf = smf[wid];
    const int nfree = lens[0];
    const int w0 = (int)(((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
    const int nw = (int)(((long long)gridDim.x * blockDim.x) >> 5);
    // packets a turn: a power of two, at most 32, fewer when that leaves warps without any
    int per = 1;
    while (per < 32 && 2 * per * nw <= nfree) per *= 2;
    const FreeBuf F = P.fr[fcur];
    const float cf = 1.0f - 2.0f / (float)P.ntc;
    int nlist = 0;
    // stage the first `cnt` members of the list
    auto stage = [&](int cnt) {
        int base = 0;
        if (lane == 0) base = atomicAdd(&lens[3], cnt);
        base = __shfl_sync(FULLMASK, base, 0);
        const long long s = (long long)base + lane;
        if (lane < cnt && s >= P.ST_cap)
            atomicOr((unsigned long long *)&P.cnt[CNT_ERR], (unsigned long long)ERRB_STAGE_CAP);
        if (lane < cnt && s < P.ST_cap) {
            const unsigned mw = mj[lane];
            const long long f = mf[lane], j = mw & 0x7ffffffu;
            const Real N = ((Real *)F.N)[f];
            const Real w = N / (Real)(int)((mw >> 27) + 1u);
            const Real d0 = ((Real *)F.dx)[f], d1 = ((Real *)F.dy)[f], d2 = ((Real *)F.dz)[f];
            const Real clk = ((Real *)F.clock)[f];
            const int nu = F.nu[f];
            // the packet's cross-section: its own mean in a shared bin, else its bin's
            const bool sgs = SH && nu == 0;
            const Real sg = sgs ? ((Real *)F.sig)[f] : Real(0);
            const int4 q = __ldg(P.q4 + j);
            const int fx = F.qx[f], fy = F.qy[f], fz = F.qz[f];
            const long long key = j * P.nf + nu;
            Real **V = (Real **)P.st_v;
            P.st_key[s] = (int)key;
            P.st_pkt[s] = (int)f;
            int bt = -1;
            if (BAR && barrier_crosses_call(P.bar[q.w], fx, fy, fz, q.x, q.y, q.z)) {
                // the share crosses the barrier: removed (counted escaped); the staged
                // contribution is empty, and the receiver side skips it
                atomicAdd(&P.esc_fx[q.w], esc_fixed(w, P, q.w));
            } else {
                Real t = (Real)(q.x - fx) * d0 + (Real)(q.y - fy) * d1 + (Real)(q.z - fz) * d2;
                Real l = t * box_unit<Real>(P, q.w);
                Real sig = sgs ? sg * (Real)P.sunit : sigma_of<Real>(P, nu);
                Real tau = (sig * ((Real *)P.nHIr)[j]) * l;
                Real A, T;
                split_absorbed<Real>(w, tau, A, T);
                bt = bin_fast<Real>(P.Rf + j * 9, P.R + j * 9, P.ax_rc, NRC, d0, d1, d2);
                V[0][s] = T;
                V[1][s] = T * (clk + light_time(l));
                V[2][s] = A;
                V[3][s] = w;
            }
            P.st_bin[s] = bt;
            P.st_rank[s] = atomicAdd(&P.seg_cnt[key], 1);
        }
        __syncwarp();
    };
    for (long long f0 = (long long)w0 * per; f0 < nfree; f0 += (long long)nw * per) {
        const long long f = f0 + lane;
        const bool on = lane < per && f < nfree;
        const bool alive = on && ((Real *)F.N)[f] > Real(0);
        Real d0 = Real(0), d1 = Real(0), d2 = Real(0);
        int qx = 0, qy = 0, qz = 0;
        if (alive) {
            d0 = ((Real *)F.dx)[f]; d1 = ((Real *)F.dy)[f]; d2 = ((Real *)F.dz)[f];
            qx = F.qx[f]; qy = F.qy[f]; qz = F.qz[f];
        }
        const float e0 = (float)d0, e1 = (float)d1, e2 = (float)d2;
        unsigned todo = __ballot_sync(FULLMASK, alive);
        bool req = false;
        // neighbour indices two packets ahead, positions one ahead
        auto index_of = [&](unsigned m) {
            return m && lane < P.kn ? F.nbr[(f0 + __ffs(m) - 1) * P.kn + lane] : 0;
        };
        int jn = index_of(todo);
        int4 qn = __ldg(P.q4 + jn);
        int jnn = index_of(todo & (todo - 1u));
        while (todo) {
            const int t = __ffs(todo) - 1;
            todo &= todo - 1u;
            const int j = jn;
            const int4 q = qn;
            jn = jnn;
            qn = __ldg(P.q4 + jn);
            jnn = index_of(todo & (todo - 1u));
            const int dx = q.x - __shfl_sync(FULLMASK, qx, t), dy = q.y - __shfl_sync(FULLMASK, qy, t),
                      dz = q.z - __shfl_sync(FULLMASK, qz, t);
            const float fx = (float)dx, fy = (float)dy, fz = (float)dz;
            const float r2 = __fmaf_rn(fx, fx, __fmaf_rn(fy, fy, fz * fz));
            const float cs = __fmaf_rn(fx, __shfl_sync(FULLMASK, e0, t),
                                       __fmaf_rn(fy, __shfl_sync(FULLMASK, e1, t),
                                                 fz * __shfl_sync(FULLMASK, e2, t))) * rsqrtf(r2);
            const bool valid = lane < P.kn && (dx | dy | dz) != 0;
            bool in = valid && cs > cf + CONE_BAND;
            const bool amb = valid && !in && !(cs < cf - CONE_BAND);
            if (__any_sync(FULLMASK, amb)) {   // inside the guard band: the exact test
                const Real x0 = __shfl_sync(FULLMASK, d0, t), x1 = __shfl_sync(FULLMASK, d1, t),
                           x2 = __shfl_sync(FULLMASK, d2, t);
                if (amb) in = cone_exact(dx, dy, dz, (double)x0, (double)x1, (double)x2, P.ntc);
            }
            const unsigned m = __ballot_sync(FULLMASK, in);
            if (!m) {
                if (lane == t) req = true;
                continue;
            }
            const int cm = __popc(m);
            if (in) {
                int p = nlist + __popc(m & ((1u << lane) - 1u));
                mj[p] = (unsigned)j | (unsigned)(cm - 1) << 27;
                mf[p] = (int)(f0 + t);
            }
            nlist += cm;
            __syncwarp();
            if (nlist >= 32) {
                stage(32);
                nlist -= 32;
                unsigned a = 0u;
                int b = 0;
                if (lane < nlist) { a = mj[32 + lane]; b = mf[32 + lane]; }
                __syncwarp();
                if (lane < nlist) { mj[lane] = a; mf[lane] = b; }
                __syncwarp();
            }
        }
        const unsigned rm = __ballot_sync(FULLMASK, req);
        if (rm) {
            int base = 0;
            if (lane == 0) base = atomicAdd(&lens[2], __popc(rm));
            base = __shfl_sync(FULLMASK, base, 0) + __popc(rm & ((1u << lane) - 1u));
            if (req && base < P.F_cap) P.req[base] = RT_FREE_BIT | (unsigned long long)f;
        }
    }
    if (nlist) stage(nlist);
}

// No accepted draw: the point on the packet's axis at h/2 (at least one quantum), rounded to
// the nearest integer offset.  FP64 path: in FP64.  FP32 path: in FP32 (fh = H/2 is exact,
// the product is rounded once), so no FP64 instruction runs in the hop loop.
__device__ __forceinline__ void axis_offset(double d0, double d1, double d2, long long H,
                                            int &Dx, int &Dy, int &Dz) {
    double fh = 0.5 * (double)H;
    if (fh < 1.0) fh = 1.0;
    Dx = (int)rint(__dmul_rn(d0, fh));
    Dy = (int)rint(__dmul_rn(d1, fh));
    Dz = (int)rint(__dmul_rn(d2, fh));
}
__device__ __forceinline__ void axis_offset(float d0, float d1, float d2, long long H,
                                            int &Dx, int &Dy, int &Dz) {
    float fh = fmaxf(0.5f * (float)(int)H, 1.0f);   // H < 2^21
    Dx = __float2int_rn(__fmul_rn(d0, fh));
    Dy = __float2int_rn(__fmul_rn(d1, fh));
    Dz = __float2int_rn(__fmul_rn(d2, fh));
}

// A virtual-particle request decoded: the packet, its sender's position and smoothing length,
// and the per-box and per-frequency values the request needs.
template <typename Real> struct VDec {
    long long h2, boff;
    unsigned long long fid, okey;
    Real N, d0, d1, d2, clk, eps, sg, sig, bu;
    float f0, f1, f2, h2f;        // the direction and the smoothing length squared in FP32
    int box, qx, qy, qz, nu, H;
};
// requests a warp takes together
#ifndef VREQ_GROUP
#define VREQ_GROUP 4
#endif

// volume, n_HI and deposit scales of a particle
__device__ __forceinline__ void vpv_load(const DevPtrs &P, long long j, float &V, float &n, float &a,
                                         float &e) {
    float4 v = ((const float4 *)P.vpv)[j];
    V = v.x; n = v.y; a = v.z; e = v.w;
}
__device__ __forceinline__ void vpv_load(const DevPtrs &P, long long j, double &V, double &n,
                                         double &a, double &e) {
    double2 v = ((const double2 *)P.vpv)[2 * j], w = ((const double2 *)P.vpv)[2 * j + 1];
    V = v.x; n = v.y; a = w.x; e = w.y;
}

// a / b, correctly rounded, for 0 < a <= b from y = the correctly rounded 1 / b (div_by_rcp);
// the plain division where the exact remainder could underflow
__device__ __forceinline__ double share_of(double a, double b, double y) {
    return a > 1e-200 && b < 1e200 ? div_by_rcp(a, b, y) : a / b;
}
__device__ __forceinline__ float share_of(float a, float b, float y) {
    if (!(a > 1e-20f && b < 1e20f)) return a / b;
    float q = __fmul_rn(a, y);
    return __fmaf_rn(__fmaf_rn(-q, b, a), y, q);
}
__device__ __forceinline__ double rcp_rn(double b) { return __drcp_rn(b); }
__device__ __forceinline__ float rcp_rn(float b) { return __frcp_rn(b); }

// Virtual particles (Sec. 2.1): a warp takes up to VREQ_GROUP consecutive requests at a time and
// passes over them in six turns, alternating between lane v serving request v (what a request
// needs once) and all lanes serving one request after the other:
//   1 lane v    decode: slot or free packet, direction, clock, identity
//   2 all       position: first accepted of 64 counter-based draws, lane = draw
//   3 lane v    escape test, cell and candidate list
//   4 all       exact kNN (rt_knn.cuh); n_HI interpolated over the neighbours, lane = neighbour
//   5 lane v    attenuation; the packet of the next hop
//   6 all       deposits, lane = neighbour
// What bounds it: instruction issue and the latency of dependent loads with FP32 packets; FP64
// (16 cycles of an SM a warp instruction) with FP64 packets.  With one request after the other
// through everything, each of the once-a-request parts took a whole warp's instructions, the
// exponential and four divisions among them; here four requests share them, and the loads of
// turn 3 and the stores of turn 5 overlap.  Measured steps against one request at a
// time with 64-bit keys: 64^3 HII region 34.6 -> 32.0 ms, the FP64 path at 32^3 19.1 -> 15.7 ms, the
// shadow test (FP64) 8.7 -> 7.8 ms.
// Work queue: every warp of the launch takes its next group from one device counter (CNT_VQ,
// zero before the hop), so all resident warps stay busy until the requests run out, whatever
// each request costs.  Results do not depend on which
// warp takes a request.
// BAR: some box has a barrier (a separate instance keeps the test out of the common case);
// SH: the shared frequency bin (likewise); IB: index bits of the exact kNN's keys (24 when a box
// holds more than 2^22 particles)
// cur, fcur: the hop's slot and free-packet buffers (launch parameters, so that buffer
// pointers are re-read from the parameter space instead of being held in registers); the
// step and hop of the random draws are read from the device counters where they are used.
template <typename Real, int NRC, bool BAR, bool SH, int IB>
__global__ void __launch_bounds__(256, VIRT_MINB(Real)) k_virtual(DevPtrs P, int cur, int fcur,
                                                                  const int *lens) {
    __shared__ VDec<Real> sdec[8][VREQ_GROUP];
    __shared__ CandQuery scell[8][VREQ_GROUP];
    __shared__ int3 spos[8][VREQ_GROUP];
    // the distances of the first 96 candidates; then the neighbours' distances, replaced by their
    // weights in the interpolated n_HI, their deposit scales and indices
    union Work {
        float f[VREQ_GROUP][96];
        struct { Real wn[VREQ_GROUP][32], ds[VREQ_GROUP][32], de[VREQ_GROUP][32]; int j[VREQ_GROUP][32]; } n;
    };
    __shared__ Work swork[8];
    __shared__ int sat[8][VREQ_GROUP][32];    // the neighbours' places in the candidate list
    __shared__ unsigned scratch[8][32];
    __shared__ unsigned sstep[2];             // step, hop << 8
    // per warp (its lane 0 keeps them): packets that go on, virtual particles outside their box,
    // and the escaped photons of one box (other boxes' are booked at once)
    __shared__ int scount[8][2], sebox[8];
    __shared__ unsigned long long sesc[8];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (threadIdx.x < 2) {
        sstep[threadIdx.x] = threadIdx.x ? cnt_word(P, CNT_HOP) << 8 : cnt_word(P, CNT_STEP);
    }
    if (threadIdx.x < 8) {
        sesc[threadIdx.x] = 0ull;
        sebox[threadIdx.x] = -1;
        scount[threadIdx.x][0] = scount[threadIdx.x][1] = 0;
    }
    __syncthreads();
    long long nreq = lens[2];
    if (nreq > P.F_cap) nreq = P.F_cap;
    const FreeBuf Fi = P.fr[fcur], Fo = P.fr[fcur ^ 1];
    VDec<Real> *mine = sdec[wid];
    unsigned long long *queue = (unsigned long long *)&P.cnt[CNT_VQ];
    const float cf = 1.0f - 2.0f / (float)P.ntc;
    // requests a warp takes at a time: fewer when few are left, so that the warps end together
    const long long nwarps = 8ll * gridDim.x;
    int grp = (int)min((long long)VREQ_GROUP, 1 + nreq / nwarps);
    // words before this lane's last adds, checked a group later (no wait for the atomics).  With
    // FP64 packets, bound by FP64 and short of instruction cache, the deposits are not unrolled and
    // a request's words are checked at the next one's.
    constexpr int DU = sizeof(Real) == 4 ? VREQ_GROUP : 1;
    unsigned long long pend_a[DU], pend_e[DU];
#pragma unroll
    for (int v = 0; v < DU; ++v) pend_a[v] = pend_e[v] = 0ull;
    bool bad = false, bad_knn = false;
    for (;;) {
        long long g0 = 0;
        if (lane == 0) g0 = (long long)atomicAdd(queue, (unsigned long long)grp);
        g0 = __shfl_sync(FULLMASK, g0, 0);
        if (g0 >= nreq) break;
        const int gn = (int)(nreq - g0 < grp ? nreq - g0 : grp);
        const long long r = g0 + lane;          // the lane's request (lane < gn)
        grp = (int)min((long long)VREQ_GROUP, 1 + (nreq - g0) / nwarps);
        // ---- 1: decode
        if (lane < gn) {
            unsigned long long code = P.req[r];
            VDec<Real> D;
            D.sg = Real(0);          // shared bin: the packet's mean cross-section (sunit)
            if (!(code & RT_FREE_BIT)) {
                Slots<Real> S(P, cur);
                long long i = (unsigned)code / (unsigned)P.S;   // slot codes < 2^31
                int s = (int)((unsigned)code % (unsigned)P.S);
                D.nu = s / NRC;
                const int4 q = P.q4[i];
                D.box = q.w;
                D.qx = q.x; D.qy = q.y; D.qz = q.z;
                D.h2 = P.h2[i];
                D.N = S.N[code];
                packet_dir(S.X[code], S.Y[code], S.Z[code], D.d0, D.d1, D.d2);
                ratios(S.C[code], S.E[code], D.N, D.clk, D.eps);
                if (SH && D.nu == 0) D.sg = ((Real *)P.slG[cur])[i * NRC + s] / D.N;
                D.okey = RT_OKEY_GEN | code;
                D.fid = gid_of(P, i, D.box) * P.S + (code - (unsigned long long)i * P.S) + 1ull;
            } else {
                long long f = (long long)(code & ~RT_FREE_BIT);
                D.box = Fi.box[f]; D.qx = Fi.qx[f]; D.qy = Fi.qy[f]; D.qz = Fi.qz[f];
                D.h2 = Fi.h2[f];
                D.N = ((Real *)Fi.N)[f];
                D.d0 = ((Real *)Fi.dx)[f]; D.d1 = ((Real *)Fi.dy)[f]; D.d2 = ((Real *)Fi.dz)[f];
                D.clk = ((Real *)Fi.clock)[f];
                D.eps = ((Real *)Fi.eps)[f];
                D.nu = Fi.nu[f];
                if (SH && D.nu == 0) D.sg = ((Real *)Fi.sig)[f];
                D.okey = Fi.okey[f] + RT_OKEY_GEN;
                D.fid = Fi.fid[f];
            }
            D.boff = P.box_off[D.box];
            D.sig = (SH && D.nu == 0) ? D.sg * (Real)P.sunit : sigma_of<Real>(P, D.nu);
            D.bu = box_unit<Real>(P, D.box);
            D.H = (int)isqrt64(D.h2);   // = floor(sqrt(h2)) exactly (h2 < 3 * 2^40), < 2^21
            D.f0 = (float)D.d0; D.f1 = (float)D.d1; D.f2 = (float)D.d2;
            D.h2f = i64_to_f(D.h2);
            mine[lane] = D;
        }
        __syncwarp();
        // ---- 2: positions
        int Dx = 0, Dy = 0, Dz = 0;             // the lane's request's offset, |D| <= H < 2^21
        bool found = false;
#pragma unroll 1
        for (int v = 0; v < gn; ++v) {
            const int H = mine[v].H;
            const unsigned span = (unsigned)(2 * H + 1);   // < 2^22
            const unsigned long long fid = mine[v].fid;
            const float f0 = mine[v].f0, f1 = mine[v].f1, f2 = mine[v].f2, h2f = mine[v].h2f;
            const uint2 key = philox_key(P.seed, 3u);
#pragma unroll 1
            for (int a0 = 0; a0 < 64; a0 += 32) {
                unsigned a = (unsigned)(a0 + lane);
                // counter: (step, hop << 8 | draw, packet id)
                uint4 u = philox4x32_10(make_uint4(sstep[0], sstep[1] | a, (unsigned)fid, (unsigned)(fid >> 32)), key);
                // floor(u * span / 2^32) - H, |e| <= H < 2^21: 32-bit integers (a 64-bit integer to
                // float conversion would run on the FP64 pipe)
                int ix = (int)__umulhi(u.x, span) - H;
                int iy = (int)__umulhi(u.y, span) - H;
                int iz = (int)__umulhi(u.z, span) - H;
                const float fx = (float)ix, fy = (float)iy, fz = (float)iz;
                const float r2 = __fmaf_rn(fx, fx, __fmaf_rn(fy, fy, fz * fz));
                const float cs = __fmaf_rn(fx, f0, __fmaf_rn(fy, f1, fz * f2)) * rsqrtf(r2);
                // inside the sphere and the cone; FP32 with guard bands (relative error of r2 below
                // 2e-7), the exact tests inside them
                bool ok = r2 > 0.0f && r2 < h2f * 0.999999f && cs > cf + CONE_BAND;
                const bool open = r2 > 0.0f && !ok && r2 < h2f * 1.000001f && !(cs < cf - CONE_BAND);
                if (__any_sync(FULLMASK, open)) {
                    if (open) {
                        long long ex = ix, ey = iy, ez = iz;
                        ok = ex * ex + ey * ey + ez * ez <= mine[v].h2 &&
                             (cs > cf + CONE_BAND ||
                              cone_exact(ix, iy, iz, (double)mine[v].d0, (double)mine[v].d1,
                                         (double)mine[v].d2, P.ntc));
                    }
                }
                unsigned m = __ballot_sync(FULLMASK, ok);
                if (m) {
                    int src = __ffs(m) - 1;
                    ix = __shfl_sync(FULLMASK, ix, src);
                    iy = __shfl_sync(FULLMASK, iy, src);
                    iz = __shfl_sync(FULLMASK, iz, src);
                    if (lane == v) { Dx = ix; Dy = iy; Dz = iz; found = true; }
                    break;
                }
            }
        }
#pragma unroll
        for (int v = 0; v < DU; ++v) bad |= pend_a[v] > (1ull << 62) || pend_e[v] > (1ull << 62);
        // ---- 3: escapes; cells
        bool alive = false;
        int gone = 0, box = 0;
        if (lane < gn) {
            const VDec<Real> &D = mine[lane];
            box = D.box;
            if (!found) axis_offset(D.d0, D.d1, D.d2, (long long)D.H, Dx, Dy, Dz);
            const int vx = D.qx + Dx, vy = D.qy + Dy, vz = D.qz + Dz;
            // outside the box: the photons escape (1); on a path through the barrier they are
            // removed, counted with the escapes (3)
            gone = (vx < 0 || vy < 0 || vz < 0 || vx >= RT_Q || vy >= RT_Q || vz >= RT_Q) ? 1
                     : (BAR && barrier_crosses_call(P.bar[box], D.qx, D.qy, D.qz, vx, vy, vz)) ? 3 : 0;
            if (gone) {
                ((Real *)Fo.N)[r] = Real(0);
            } else {
                alive = true;
                spos[wid][lane] = make_int3(vx, vy, vz);
                scell[wid][lane] = cand_query(P.grid, box, vx, vy, vz);
            }
        }
        const unsigned am = __ballot_sync(FULLMASK, alive), gm = __ballot_sync(FULLMASK, gone != 0);
        if (gm) {
            int eb = sebox[wid];
            if (eb < 0) eb = __shfl_sync(FULLMASK, box, __ffs(gm) - 1);
            unsigned long long es = gone ? esc_fixed(mine[lane & (VREQ_GROUP - 1)].N, P, box) : 0ull;
            if (gone && box != eb) {
                atomicAdd(&P.esc_fx[box], es);
                es = 0ull;
            }
#pragma unroll
            for (int o = 1; o < VREQ_GROUP; o <<= 1) es += __shfl_xor_sync(FULLMASK, es, o);
            const int out = __popc(__ballot_sync(FULLMASK, gone == 1));
            __syncwarp();
            if (lane == 0) {
                sebox[wid] = eb;
                sesc[wid] += es;
                scount[wid][1] += out;
            }
        }
        __syncwarp();
        // ---- 4: neighbours and n_HI.  Loads of all four requests side by side: the candidates'
        // distances; after the order of each, the neighbours and their properties
        Work &W = swork[wid];
        const bool valid = lane < P.kn;
#pragma unroll
        for (int v = 0; v < VREQ_GROUP; ++v) {
            if (!((am >> v) & 1u)) continue;
            const int3 q = spos[wid][v];
            const float4 *items = scell[wid][v].items;
            const unsigned *cd = P.grid.cand + scell[wid][v].a;
            const int len = scell[wid][v].len;
#pragma unroll
            for (int b = 0; b < 3; ++b)
                if (lane + 32 * b < len)
                    W.f[v][lane + 32 * b] = cand_dist(items, __ldg(cd + lane + 32 * b), (float)q.x,
                                                      (float)q.y, (float)q.z);
        }
#pragma unroll 1
        for (unsigned m = am; m; m &= m - 1u) {
            const int v = __ffs(m) - 1;
            const int3 q = spos[wid][v];
            const CandQuery Q = scell[wid][v];
            int at;
            if (!cand_order(W.f[v][lane], W.f[v][lane + 32], W.f[v][lane + 64], Q.items, P.grid.cand + Q.a,
                            Q.len, (float)q.x, (float)q.y, (float)q.z, Q.rq_up, Q.w, P.kn, scratch[wid],
                            at)) {
                KnnOut o = knn_exact_query<IB>(grid_of_box(P.grid, mine[v].box), P.grid.cand, Q.a,
                                               Q.a + Q.len, Q.rq_up, Q.w, q.x, q.y, q.z, P.kn,
                                               (int *)scratch[wid]);
                // a k-th neighbour beyond the key range: reported; indices kept inside the box
                if (!o.ok) bad_knn = true;
                const int box = mine[v].box;
                if (o.idx < 0 || o.idx >= P.box_off[box + 1] - mine[v].boff) o.idx = 0;
                at = o.idx | INT_MIN;
            }
            sat[wid][v][lane] = at;
        }
        __syncwarp();
        Real msw = Real(1), mswn = Real(0);
        long long mh2v = 0;
        float4 it[VREQ_GROUP];
#pragma unroll
        for (int v = 0; v < VREQ_GROUP; ++v) {
            it[v] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (!((am >> v) & 1u) || !valid) continue;
            const int at = sat[wid][v][lane];
            if (at >= 0) {
                it[v] = __ldg(scell[wid][v].items + (__ldg(P.grid.cand + scell[wid][v].a + at) & 0xffffffu));
            } else {   // (the exact search gives the particle)
                const int i = at & INT_MAX;
                const int4 p = __ldg(P.q4 + mine[v].boff + i);
                it[v] = make_float4((float)p.x, (float)p.y, (float)p.z, __int_as_float(i));
            }
        }
#pragma unroll
        for (int v = 0; v < VREQ_GROUP; ++v) {
            if (!((am >> v) & 1u)) continue;
            const int3 q = spos[wid][v];
            const long long kd2 = exact_d2(it[v], (float)q.x, (float)q.y, (float)q.z);
            const long long h2v = __shfl_sync(FULLMASK, kd2, P.kn - 1);
            if (IB != KNN_IB_SMALL && h2v >= knn_d2max<IB>()) bad_knn = true;
            if (lane == v) mh2v = h2v;
            W.n.wn[v][lane] = to_real<Real>(kd2);
            W.n.j[v][lane] = (int)(mine[v].boff + __float_as_int(it[v].w));
        }
        // (a lane reads back its own words)
        Real Vn = Real(0), nn = Real(0), dsn = Real(0), den = Real(0);
        if (am && valid) vpv_load(P, W.n.j[__ffs(am) - 1][lane], Vn, nn, dsn, den);
#pragma unroll 1
        for (unsigned m = am; m; m &= m - 1u) {
            const int v = __ffs(m) - 1;
            const Real Vj = Vn, nhj = nn;
            W.n.ds[v][lane] = dsn;
            W.n.de[v][lane] = den;
            const unsigned m2 = m & (m - 1u);   // the next request's neighbours, loaded ahead
            if (m2 && valid) vpv_load(P, W.n.j[__ffs(m2) - 1][lane], Vn, nn, dsn, den);
            const Real kr = W.n.wn[v][lane], hr = __shfl_sync(FULLMASK, kr, P.kn - 1);
            Real om = Real(0);
            if (valid) {
                Real qq = hr > Real(0) ? rt_sqrt<Real>(kr / hr) : Real(0);
                om = Vj * kernel_w<Real>(qq);
                Fo.nbr[(g0 + v) * P.kn + lane] = W.n.j[v][lane];
            }
            Real sw = om;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sw += __shfl_xor_sync(FULLMASK, sw, o);
            if (!(sw > Real(0))) {
                om = valid ? Vj : Real(0);
                sw = om;
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) sw += __shfl_xor_sync(FULLMASK, sw, o);
            }
            const Real wn = valid ? om * nhj : Real(0);
            Real sn = wn;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) sn += __shfl_xor_sync(FULLMASK, sn, o);
            W.n.wn[v][lane] = wn;
            if (lane == v) { msw = sw; mswn = sn; }
        }
        // ---- 5: attenuation; the packet of the next hop
        Real A = Real(0), ry = Real(0);
        bool on = false;
        if (alive) {
            const VDec<Real> &D = mine[lane];
            const Real nHIv = mswn / msw;
            const Real t = (Real)Dx * D.d0 + (Real)Dy * D.d1 + (Real)Dz * D.d2;
            const Real l = t * D.bu;
            const Real tau = (D.sig * nHIv) * l;
            Real T;
            split_absorbed<Real>(D.N, tau, A, T);
            ry = rcp_rn(mswn);
            on = T > Real(0);
            Fo.box[r] = D.box;
            Fo.qx[r] = D.qx + Dx; Fo.qy[r] = D.qy + Dy; Fo.qz[r] = D.qz + Dz;
            Fo.h2[r] = mh2v;
            ((Real *)Fo.N)[r] = T;
            ((Real *)Fo.dx)[r] = D.d0; ((Real *)Fo.dy)[r] = D.d1; ((Real *)Fo.dz)[r] = D.d2;
            ((Real *)Fo.clock)[r] = D.clk + light_time(l);
            ((Real *)Fo.eps)[r] = D.eps;
            if (SH && D.nu == 0) ((Real *)Fo.sig)[r] = D.sg;
            Fo.nu[r] = D.nu;
            Fo.okey[r] = D.okey;
            Fo.fid[r] = mix64(D.fid);
        }
        const int non = __popc(__ballot_sync(FULLMASK, on));
        if (lane == 0) scount[wid][0] += non;
        // ---- 6: deposits
#pragma unroll DU
        for (int v = 0; v < VREQ_GROUP; ++v) {
            const int ps = DU == 1 ? 0 : v;
            if (DU == 1) bad |= pend_a[0] > (1ull << 62) || pend_e[0] > (1ull << 62);
            pend_a[ps] = 0ull;
            pend_e[ps] = 0ull;
            if (!((am >> v) & 1u)) continue;
            const Real Av = __shfl_sync(FULLMASK, A, v), sn = __shfl_sync(FULLMASK, mswn, v),
                       y = __shfl_sync(FULLMASK, ry, v);
            const Real wn = W.n.wn[v][lane];
            if (valid && sn > Real(0) && wn > Real(0)) {
                const long long j = W.n.j[v][lane];
                const Real dsj = W.n.ds[v][lane], dej = W.n.de[v][lane];
                const Real Ak = Av * share_of(wn, sn, y);
                const long long key2 = j * P.nf + mine[v].nu;
                // two fixed-point words: units of 2^-40 N_HI and 2^-72 N_HI (integer sums do not
                // depend on their order)
                const Real fa = Ak * dsj;
                const Real fe = Ak * mine[v].eps * dej;
                if (fa > Real(0)) {
                    unsigned long long qh = 0, ql = 0;
                    bad |= !fx_split(fa, qh, ql);
                    if (qh) pend_a[ps] = atomicAdd(&P.fx_abs[key2], qh);
                    if (ql) atomicAdd(&P.fx_lo[key2], ql);
                }
                if (fe > Real(0)) {
                    bad |= fe > Real(4.0e18);
                    pend_e[ps] = atomicAdd(&P.fx_E[key2], to_fixed(fe));
                }
            }
        }
        __syncwarp();   // the group's shared values are read before the next group's are written
    }
#pragma unroll
    for (int v = 0; v < DU; ++v) bad |= pend_a[v] > (1ull << 62) || pend_e[v] > (1ull << 62);
    if (bad) atomicOr((unsigned long long *)&P.cnt[CNT_ERR], (unsigned long long)ERRB_RANGE);
    if (bad_knn) atomicOr((unsigned long long *)&P.cnt[CNT_ERR], (unsigned long long)ERRB_KNN);
    __syncthreads();
    if (lane == 0 && sesc[wid]) atomicAdd(&P.esc_fx[sebox[wid]], sesc[wid]);
    if (threadIdx.x < 2) {
        int t = 0;
        for (int k = 0; k < 8; ++k) t += scount[k][threadIdx.x];
        if (t) atomicAdd((unsigned long long *)&P.cnt[threadIdx.x ? CNT_VESC : CNT_LIVE], (unsigned long long)t);
    }
}

// The receiver groups with work this hop: receivers touched by a gas sender, receivers of
// staged free-packet contributions, and particles holding waiting packets.  Four consecutive
// keys a thread (16-byte loads); block-level compaction with one atomic per block; the order of
// the list does not matter.  An entry is the key, with bit 31 set when a gas sender touched it
// (the flag is cleared here).  A group with staged contributions gets its segment of the list
// of staged contributions here, from one counter (lens[5]).  The next slot buffer's occupancy
// and activity words are cleared here for the receiver side.
__global__ void __launch_bounds__(256) k_worklist(DevPtrs P, int cur, int *lens) {
    __shared__ int wcount[8], wbase[8];
    const long long nkey = P.n * P.nf;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    for (long long k0 = (long long)blockIdx.x * 1024; k0 < nkey; k0 += (long long)gridDim.x * 1024) {
        const long long key = k0 + 4 * threadIdx.x;
        unsigned fl = 0u, tf = 0u;            // four flags: with work; touched
        int4 sc = make_int4(0, 0, 0, 0);      // staged contributions
        if (key < nkey) {   // (the arrays are padded to whole fours, with zeros)
            const uchar4 t = *(const uchar4 *)(P.touched + key);
            const int4 c = *(const int4 *)(P.seg_cnt + key);
            const uint4 o = *(const uint4 *)(P.occ[cur] + key), a = *(const uint4 *)(P.act[cur] + key);
            tf = (t.x ? 1u : 0u) | (t.y ? 2u : 0u) | (t.z ? 4u : 0u) | (t.w ? 8u : 0u);
            fl = tf | (c.x || (o.x & ~a.x) ? 1u : 0u) | (c.y || (o.y & ~a.y) ? 2u : 0u) |
                 (c.z || (o.z & ~a.z) ? 4u : 0u) | (c.w || (o.w & ~a.w) ? 8u : 0u);
            if (tf) *(uchar4 *)(P.touched + key) = make_uchar4(0, 0, 0, 0);
            *(uint4 *)(P.occ[cur ^ 1] + key) = make_uint4(0u, 0u, 0u, 0u);
            *(uint4 *)(P.act[cur ^ 1] + key) = make_uint4(0u, 0u, 0u, 0u);
            sc = c;
        }
        const int st = sc.x + sc.y + sc.z + sc.w;
        if (__any_sync(FULLMASK, st != 0)) {
            const int incl = (int)lane_scan((unsigned)st);
            int so = 0;
            if (lane == 31) so = atomicAdd(&lens[5], incl);
            so = __shfl_sync(FULLMASK, so, 31) + incl - st;
            if (sc.x) P.seg_off[key] = so;
            if (sc.y) P.seg_off[key + 1] = so + sc.x;
            if (sc.z) P.seg_off[key + 2] = so + sc.x + sc.y;
            if (sc.w) P.seg_off[key + 3] = so + sc.x + sc.y + sc.z;
        }
        if (!__syncthreads_or(fl != 0u)) continue;
        const unsigned incl = lane_scan((unsigned)__popc(fl));
        if (lane == 31) wcount[w] = (int)incl;
        __syncthreads();
        if (threadIdx.x == 0) {
            int t = 0;
            for (int k = 0; k < 8; ++k) { wbase[k] = t; t += wcount[k]; }
            int b = atomicAdd(&lens[4], t);
            for (int k = 0; k < 8; ++k) wbase[k] += b;
        }
        __syncthreads();
        int p = wbase[w] + (int)incl - __popc(fl);
        for (unsigned x = fl; x; x &= x - 1u) {
            int q = __ffs(x) - 1;
            P.worklist[p++] = (int)((unsigned)(key + q) | ((tf >> q) & 1u ? 0x80000000u : 0u));
        }
        __syncthreads();
    }
}

// the staged contributions into their receivers' segments, with the order of their packets
__global__ void __launch_bounds__(256) k_seg_fill(DevPtrs P, int fcur, const int *lens) {
    long long nst = lens[3];
    if (nst > P.ST_cap) nst = P.ST_cap;
    for (long long s = (long long)blockIdx.x * blockDim.x + threadIdx.x; s < nst;
         s += (long long)gridDim.x * blockDim.x) {
        const int key = P.st_key[s], rank = P.st_rank[s], f = P.st_pkt[s];
        const unsigned long long order = P.fr[fcur].okey[f];   // (loaded beside the offset)
        const int pos = P.seg_off[key] + rank;
        P.seg_ent[pos] = make_int2((int)s, f);
        P.seg_key[pos] = order;
    }
}

// absorptions of one receiver group in one hop.  FP64 path: FP64 sums.  FP32 path: the
// group's (fixed-order) sums go into the particle's fixed-point words, like the virtual-particle
// deposits, so no FP64 instruction runs in the hop loop; pass counts stay in FP32.  Returns the
// high absorption word before the add (0 on the FP64 path), which the caller range-checks one
// group later, so that the group does not wait for the atomic's round trip.
template <typename Real>
__device__ __forceinline__ unsigned long long deposit_group(const DevPtrs &P, long long key,
                                                            long long j, int box, Real a, Real ae,
                                                            Real w);
template <>
__device__ __forceinline__ unsigned long long deposit_group<double>(const DevPtrs &P,
                                                                    long long key, long long j,
                                                                    int box, double a, double ae,
                                                                    double w) {
    double nm = P.norm[box];
    P.abs[key] += a * nm;
    P.absE[key] += ae * nm * P.eunit;
    P.pass[key] += w * nm;
    return 0ull;
}
template <>
__device__ __forceinline__ unsigned long long deposit_group<float>(const DevPtrs &P,
                                                                   long long key, long long j,
                                                                   int box, float a, float ae,
                                                                   float w) {
    // atomics: virtual-particle deposits into the same words may run at the same time
    unsigned long long old = 0ull;
    float fa = a * pv<float>(P, j, PV_DEP);
    if (fa > 0.0f) {
        unsigned long long qh, ql;
        if (fx_split(fa, qh, ql)) {
            old = atomicAdd(&P.fx_abs[key], qh);
            atomicAdd(&P.fx_lo[key], ql);
        } else {
            atomicOr((unsigned long long *)&P.cnt[CNT_ERR], (unsigned long long)ERRB_RANGE);
        }
    }
    float fe = ae * pv<float>(P, j, PV_DEPE);
    if (fe > 0.0f) atomicAdd(&P.fx_E[key], f2u64_rz(fe + 0.5f));
    P.passf[key] += w;
    return old;
}

// What the receiver side keeps of one contribution, in pairs: (T, T d0), (T d1, T d2),
// (T clock, T eps), (A, A eps), and w with, in a shared frequency bin, T sigma.
#define BV_N 5

// One gas contribution to receiver j in frequency nu: reverse edge e, bit b of its word.
// Attenuates, stores the values in sv[.][lane] and returns its reception cone, or -1 when a
// barrier removed it (counted escaped).
template <typename Real, int G, bool BAR, bool SH>
__device__ __forceinline__ int gas_contribution(const DevPtrs &P, long long e, int b, long long j,
                                                int nu, int box, Real u, Real sig_nhi,
                                                Pair<Real> (*sv)[32], int lane) {
    float4 ed = __ldg(P.rev4 + e);
    bool sgs = SH && nu == 0;
    Real w, d0, d1, d2, clk, eps, sgc = Real(0);
    rec_load(P.rec, (long long)__float_as_int(ed.w) * P.S + (long long)nu * G + b, w, d0, d1, d2,
             clk, eps, sgs, sgc);
    if (BAR) {
        const int4 q = P.q4[j];
        if (barrier_crosses_call(P.bar[box], q.x - (int)ed.x, q.y - (int)ed.y, q.z - (int)ed.z, q.x,
                                 q.y, q.z)) {
            atomicAdd(&P.esc_fx[box], esc_fixed(w, P, box));
            return -1;
        }
    }
    Real t = (Real)ed.x * d0 + (Real)ed.y * d1 + (Real)ed.z * d2;
    Real l = t * u;
    Real A, T;
    // in a shared bin each packet carries its own mean cross-section
    Real sn = sgs ? (sgc * (Real)P.sunit) * ((Real *)P.nHIr)[j] : sig_nhi;
    split_absorbed<Real>(w, sn * l, A, T);
    sv[0][lane] = make_pair2(T, T * d0);
    sv[1][lane] = make_pair2(T * d1, T * d2);
    sv[2][lane] = make_pair2(T * (clk + light_time(l)), T * eps);
    sv[3][lane] = make_pair2(A, A * eps);
    sv[4][lane] = make_pair2(w, sgs ? T * sgc : Real(0));
    return bin_fast<Real>(P.Rf + j * 9, P.R + j * 9, P.ax_rc, G, d0, d1, d2);
}

// A staged contribution (e.x) of a packet (e.y) of free buffer fcur: its values into sv[.][lane], its cone
// (-1: removed).
template <typename Real, bool SH>
__device__ __forceinline__ int staged_contribution(const DevPtrs &P, int fcur, int2 e, int nu,
                                                   Pair<Real> (*sv)[32], int lane) {
    Real *const *V = (Real *const *)P.st_v;
    const int s = e.x, f = e.y, bin = P.st_bin[s];
    if (bin >= 0) {
        const FreeBuf &F = P.fr[fcur];
        const Real T = V[0][s], A = V[2][s], eps = ((Real *)F.eps)[f];
        sv[0][lane] = make_pair2(T, T * ((Real *)F.dx)[f]);
        sv[1][lane] = make_pair2(T * ((Real *)F.dy)[f], T * ((Real *)F.dz)[f]);
        sv[2][lane] = make_pair2(V[1][s], T * eps);
        sv[3][lane] = make_pair2(A, A * eps);
        sv[4][lane] = make_pair2(V[3][s], SH && nu == 0 ? T * ((Real *)F.sig)[f] : Real(0));
    }
    return bin;
}

// A segment of n > 8 contributions brought into packet order by the whole warp: blocks of 32 by
// counting earlier packets (distinct), then sorted runs merged in pairs, an entry's place being its
// place in its run and the earlier ones of the other (binary search).  The passes alternate
// between ent and tmp and end in ent.  Counting the earlier packets of the whole segment, without
// the merges, is quadratic: 20,000 sources within one smoothing length give their neighbours
// segments of 20,000, and a step of a 32^3 box took 2.1 s (FP32), 35 ms now; with 4,096 sources 96
// and 9 ms.
__device__ void order_wide(const unsigned long long *okey, int2 *ent, int2 *tmp, unsigned n) {
    const unsigned lane = threadIdx.x & 31u;
    bool odd = false;                  // number of merge passes
    for (unsigned L = 32; L < n; L *= 2) odd = !odd;
    int2 *a = odd ? tmp : ent, *b = odd ? ent : tmp;
    for (unsigned c = 0; c < n; c += 32) {
        const bool on = c + lane < n;
        const int2 s = on ? ent[c + lane] : make_int2(0, 0);
        const unsigned long long key = on ? okey[s.y] : ~0ull;
        int r = 0;
        for (int k = 0; k < 32; ++k) r += __shfl_sync(FULLMASK, key, k) < key;
        if (on) a[c + r] = s;
    }
    __syncwarp();
    for (unsigned L = 32; L < n; L *= 2) {
        for (unsigned t = lane; t < n; t += 32) {
            const int2 s = a[t];
            const unsigned long long key = okey[s.y];
            const unsigned run = t & ~(L - 1u), other = run ^ L;
            unsigned lo = min(other, n), hi = min(other + L, n);
            const unsigned o0 = lo;
            while (lo < hi) {
                const unsigned m = (lo + hi) >> 1;
                if (okey[a[m].y] < key) lo = m + 1u;
                else hi = m;
            }
            b[min(run, other) + (t - run) + (lo - o0)] = s;
        }
        __syncwarp();
        int2 *x = a;
        a = b;
        b = x;
    }
}

// the four segments of a warp (n contributions each, lanes of eight hold the same): those of more
// than eight, one after the other
static __device__ __noinline__ void order_long(const unsigned long long *okey, int2 *ent, int2 *tmp,
                                               int n) {
    for (unsigned w = __ballot_sync(FULLMASK, n > 8 && (threadIdx.x & 7) == 0); w; w &= w - 1u) {
        const int k = __ffs(w) - 1;
        order_wide(okey, (int2 *)__shfl_sync(FULLMASK, (unsigned long long)ent, k),
                   (int2 *)__shfl_sync(FULLMASK, (unsigned long long)tmp, k),
                   (unsigned)__shfl_sync(FULLMASK, n, k));
    }
}

// those of up to eight, all at once: a lane an entry.  Out of line: few groups have any, and inlined
// it costs the receiver side registers.
static __device__ __noinline__ void order_segments(const unsigned long long *key, int2 *ent, int n) {
    const int l = threadIdx.x & 7;
    const bool on = n <= 8 && l < n;
    const int2 s = on ? ent[l] : make_int2(0, 0);
    const unsigned long long v = on ? key[l] : ~0ull;
    int r = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) r += __shfl_sync(FULLMASK, v, k, 8) < v;
    if (on) ent[r] = s;
    __syncwarp();
}

// the merged packet of one reception cone: N, N d, N clock, N eps (and N sigma, shared bin)
template <typename Real, bool SH> struct ConeSum {
    KSum2<Real> NX, YZ, CE;
    KSum<Real> G;
    __device__ __forceinline__ void zero() {
        NX.init(Real(0), Real(0)); YZ.init(Real(0), Real(0)); CE.init(Real(0), Real(0));
        G.init(Real(0));
    }
    __device__ __forceinline__ void add(Pair<Real> (*sv)[32], int t, bool sgs) {
        NX.add(sv[0][t]); YZ.add(sv[1][t]); CE.add(sv[2][t]);
        if (sgs) G.add(sv[4][t].y);
    }
    // a packet that waited in the cone
    __device__ __forceinline__ void load(const Slots<Real> &S, const Real *SG, long long s,
                                         long long g, bool sgs) {
        NX.init(S.N[s], S.X[s]); YZ.init(S.Y[s], S.Z[s]); CE.init(S.C[s], S.E[s]);
        G.init(sgs ? SG[g] : Real(0));
    }
    __device__ __forceinline__ Real photons() const { return NX.get().x; }
    __device__ __forceinline__ Real clock() const { return CE.get().x; }
    __device__ __forceinline__ void store(const Slots<Real> &S, Real *SG, long long s, long long g,
                                          bool sgs) const {
        const Pair<Real> a = NX.get(), b = YZ.get(), c = CE.get();
        S.N[s] = a.x; S.X[s] = a.y; S.Y[s] = b.x; S.Z[s] = b.y; S.C[s] = c.x; S.E[s] = c.y;
        if (sgs) SG[g] = G.get();
    }
};

// the absorption sums of a group: A, A eps, w
template <typename Real> struct AbsSum {
    KSum2<Real> A;
    KSum<Real> W;
    __device__ __forceinline__ void zero() {
        A.init(Real(0), Real(0));
        W.init(Real(0));
    }
    __device__ __forceinline__ void add(Pair<Real> (*sv)[32], int t) {
        A.add(sv[3][t]);
        W.add(sv[4][t].x);
    }
};

// number of set bits of each byte
__device__ __forceinline__ unsigned byte_popc(unsigned x) {
    x = x - ((x >> 1) & 0x55555555u);
    x = (x & 0x33333333u) + ((x >> 2) & 0x33333333u);
    return (x + (x >> 4)) & 0x0f0f0f0fu;
}
// One receiver group of 32 cones by a whole warp, lane = reception cone, whatever its number of
// edges, contributions and waiting packets: edges 32 at a time, contributions 32 at a time,
// each cone's lane adding its contributions in list order.
template <typename Real, bool BAR, bool SH>
__device__ __forceinline__ void wide_group(const DevPtrs &P, int cur, int fcur, long long key,
                                           bool touched, int fc, int so, Pair<Real> (*sv)[32], unsigned *list,
                                           unsigned *smask, unsigned long long &pend, bool &bad,
                                           int *stot) {
    const int lane = threadIdx.x & 31;
    const int j = (int)((unsigned)key / (unsigned)P.nf), nu = (int)((unsigned)key % (unsigned)P.nf);
    const int box = P.pbox[j];
    const unsigned park = P.occ[cur][key] & ~P.act[cur][key];
    const bool sgs = SH && nu == 0;
    const long long sidx = (long long)j * P.S + (long long)nu * 32 + lane;
    const long long gidx = (long long)j * 32 + lane;
    ConeSum<Real, SH> a;
    a.zero();
    if ((park >> lane) & 1u) a.load(Slots<Real>(P, cur), (const Real *)P.slG[cur], sidx, gidx, sgs);
    AbsSum<Real> ab;
    ab.zero();
    auto merge = [&](int bin) {
        smask[lane] = 0u;
        __syncwarp();
        if (bin >= 0) {
            atomicOr(&smask[bin], 1u << lane);
            ab.add(sv, lane);
        }
        __syncwarp();
        unsigned m = smask[lane];
        while (m) {
            int t = __ffs(m) - 1;
            m &= m - 1u;
            a.add(sv, t, sgs);
        }
        __syncwarp();
    };
    if (touched) {
        const Real u = box_unit<Real>(P, box);
        const Real sig_nhi = sigma_of<Real>(P, nu) * ((Real *)P.nHIr)[j];
        const int e0 = P.rev_off[j], e1 = P.rev_off[j + 1];
        unsigned *bmr = P.bm + (long long)nu * P.n * P.kn;
        for (int eb = e0; eb < e1; eb += 32) {
            unsigned word = 0u;
            if (eb + lane < e1) {
                word = bmr[eb + lane];
                if (word) bmr[eb + lane] = 0u;
            }
            const unsigned cw = (unsigned)__popc(word);
            const unsigned incl = lane_scan(cw);
            const int total = (int)__shfl_sync(FULLMASK, incl, 31);
            for (int cb = 0; cb < total; cb += 32) {
                int p = (int)(incl - cw) - cb;
                for (unsigned x = word; x; x &= x - 1u, ++p)
                    if (p >= 0 && p < 32) list[p] = (unsigned)(__ffs(x) - 1) | (unsigned)lane << 5;
                __syncwarp();
                const bool has = cb + lane < total;
                const unsigned code = has ? list[lane] : 0u;
                int bin = -1;
                if (has)
                    bin = gas_contribution<Real, 32, BAR, SH>(P, (long long)eb + (code >> 5), code & 31u, j,
                                                              nu, box, u, sig_nhi, sv, lane);
                merge(bin);
            }
        }
    }
    for (int cb = 0; cb < fc; cb += 32) {
        int bin = -1;
        if (cb + lane < fc)
            bin = staged_contribution<Real, SH>(P, fcur, P.seg_ent[so + cb + lane], nu, sv, lane);
        merge(bin);
    }
    const Real N = a.photons();
    const bool occ = N > Real(0);
    const bool act = occ && (a.clock() / N < (Real)P.dt);
    const unsigned bo = __ballot_sync(FULLMASK, occ), ba = __ballot_sync(FULLMASK, act);
    if (occ) a.store(Slots<Real>(P, cur ^ 1), (Real *)P.slG[cur ^ 1], sidx, gidx, sgs);
    Real av = ab.A.get().x, ae = ab.A.get().y, w = ab.W.get();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        av += __shfl_down_sync(FULLMASK, av, o);
        ae += __shfl_down_sync(FULLMASK, ae, o);
        w += __shfl_down_sync(FULLMASK, w, o);
    }
    if (lane == 0) {
        P.occ[cur ^ 1][key] = bo;
        P.act[cur ^ 1][key] = ba;
        atomicAdd(&stot[0], __popc(bo));
        atomicAdd(&stot[1], __popc(ba));
        if (touched || fc > 0) {
            bad |= pend > (1ull << 62);
            pend = deposit_group<Real>(P, key, j, box, av, ae, w);
        }
    }
}

// Receiver side.  A warp takes four receiver groups (particle j, frequency nu) of the work list
// at a time, expands the bitmap bits of their reverse edges into one list of contributions, and
// computes 32 contributions of that list at a time, one per lane: gathering a sender's record,
// attenuation, reception cone.  Then the contributions are merged in their fixed order (sender,
// slot; staged ones after them in packet order): the lane owning a target cone adds them.
// What bounds it: instructions and the latency of the gathers.  A group has few contributions
// (8.6 with 8 cones behind a fast front, 3.8 with 32 cones in the HII region), so a group of
// n_rc lanes of its own left most lanes idle in the long part, the contributions
// (13.6 of 32 active); four groups share a pass here.  Measured per step against a
// group of n_rc lanes each: 64^3 HII region, 32 cones, 17.5 -> 10.7 ms, the FP64 path at 32^3
// 6.8 -> 3.5 ms; 2.1 M particles behind a fast front, 8 cones, 189 -> 132 ms.
//   8 cones: lane = (group, cone), so the four groups' 32 cones stay in registers whatever the
//   number of contributions.
//   32 cones: groups of at most 32 contributions in all are merged together, the lowest lane of
//   each (group, cone) adding; a group of more (or of waiting packets, or of more than 64
//   edges) has enough work for a warp of its own (wide_group).
// Each sum keeps the order and the tree that one lane per cone and contribution gives: the
// absorption sums of a group are Kahan sums per lane (position of the contribution in its run
// of n_rc edges, modulo n_rc), then a tree over the lanes.  Results do not depend on how
// groups meet in a warp.
// Groups come from the work list; the next buffer's occupancy words were cleared by the
// work-list kernel.  cur, fcur: the slot and free-packet buffers holding the hop's packets.
template <typename Real, int G, bool BAR, bool SH>
__global__ void __launch_bounds__(256, HOP_MINB(Real)) k_phaseB(DevPtrs P, int cur, int fcur,
                                                                const int *lens) {
    __shared__ Pair<Real> svs[8][BV_N][32];
    __shared__ unsigned slist[8][32];
    __shared__ unsigned smask[8][2][32];
    __shared__ int snext;
    __shared__ int stot[2];            // the block's packets written, and those able to move
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    Pair<Real> (*sv)[32] = svs[wid];
    unsigned *list = slist[wid];
    const int kq = lane >> 3;                  // the lane's group of the four
    const int nxt = cur ^ 1;
    // each block takes one contiguous chunk of the work list, in fours; its warps pull from it
    // through a shared counter, so that they finish together
    long long ng = lens[4];
    long long chunk = ((ng + gridDim.x - 1) / gridDim.x + 3) & ~3ll;
    long long gb0 = (long long)blockIdx.x * chunk;
    long long gb1 = gb0 + chunk < ng ? gb0 + chunk : ng;
    if (threadIdx.x == 0) snext = stot[0] = stot[1] = 0;
    __syncthreads();
    unsigned long long pend = 0ull;   // the high absorption word before the last deposit
    bool bad = false;
    for (;;) {
        long long g0 = 0;
        if (lane == 0) g0 = gb0 + atomicAdd(&snext, 4);
        g0 = __shfl_sync(FULLMASK, g0, 0);
        if (g0 >= gb1) break;
        // the group of each eight lanes
        const bool kv = g0 + kq < gb1;
        const unsigned wv = kv ? (unsigned)P.worklist[g0 + kq] : 0u;
        const long long key = wv & 0x7fffffffu;
        const bool touched = (wv >> 31) != 0u;
        const int j = (int)((unsigned)key / (unsigned)P.nf);
        const int nu = (int)((unsigned)key % (unsigned)P.nf);
        const unsigned park = kv ? P.occ[cur][key] & ~P.act[cur][key] : 0u;
        const int fc = kv ? P.seg_cnt[key] : 0;
        const int so = fc > 0 ? P.seg_off[key] : 0;
        const int e0 = touched ? P.rev_off[j] : 0;
        const int ne = touched ? P.rev_off[j + 1] - e0 : 0;
        const int box = P.pbox[j];
        const Real u = box_unit<Real>(P, box);
        const Real sig_nhi = sigma_of<Real>(P, nu) * ((Real *)P.nHIr)[j];
        Slots<Real> So(P, cur), Sn(P, nxt);
        if (__any_sync(FULLMASK, fc > 0)) {
            order_segments(P.seg_key + so, P.seg_ent + so, fc);
            if (__any_sync(FULLMASK, fc > 8))
                order_long(P.fr[fcur].okey, P.seg_ent + so, P.seg_tmp + so, fc);
            if ((lane & 7) == 0 && fc > 0) P.seg_cnt[key] = 0;   // for the next hop
        }
        // a group's values to the lanes that work on it
        auto of = [&](auto v, int k) { return __shfl_sync(FULLMASK, v, 8 * k); };
        if constexpr (G == 8) {
            const int bl = lane & 7;
            const long long sidx = (long long)j * P.S + (long long)nu * G + bl;
            const long long gidx = (long long)j * G + bl;
            const bool sgs = SH && nu == 0;
            ConeSum<Real, SH> a;
            a.zero();
            if ((park >> bl) & 1u) a.load(So, (const Real *)P.slG[cur], sidx, gidx, sgs);
            AbsSum<Real> ab;
            ab.zero();
            // merge the contributions of the lanes: group kk, cone bin (-1: none), and the lane
            // ol of the group's absorption sums
            auto merge = [&](int kk, int bin, int ol) {
                smask[wid][0][lane] = 0u;
                smask[wid][1][lane] = 0u;
                __syncwarp();
                if (bin >= 0) {
                    atomicOr(&smask[wid][0][8 * kk + bin], 1u << lane);
                    atomicOr(&smask[wid][1][8 * kk + ol], 1u << lane);
                }
                __syncwarp();
                unsigned m = smask[wid][0][lane], m2 = smask[wid][1][lane];
                while (m) {
                    int t = __ffs(m) - 1;
                    m &= m - 1u;
                    a.add(sv, t, sgs);
                }
                while (m2) {
                    int t = __ffs(m2) - 1;
                    m2 &= m2 - 1u;
                    ab.add(sv, t);
                }
                __syncwarp();
            };
            const int nemax = __reduce_max_sync(FULLMASK, ne);
            for (int eb = 0; eb < nemax; eb += 64) {
                // lane: edges 2 lane and 2 lane + 1 of the block; the four groups' words, eight
                // bits each, in one register per edge
                unsigned w0[4], w1[4];
                unsigned *bw[4];
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    int rem = of(ne, kk) - eb - 2 * lane;
                    bw[kk] = P.bm + (long long)of(nu, kk) * P.n * P.kn + of(e0, kk) + eb + 2 * lane;
                    w0[kk] = rem > 0 ? bw[kk][0] : 0u;
                    w1[kk] = rem > 1 ? bw[kk][1] : 0u;
                }
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    if (w0[kk]) bw[kk][0] = 0u;
                    if (w1[kk]) bw[kk][1] = 0u;
                }
                const unsigned W0 = w0[0] | w0[1] << 8 | w0[2] << 16 | w0[3] << 24;
                const unsigned W1 = w1[0] | w1[1] << 8 | w1[2] << 16 | w1[3] << 24;
                // positions in the list (group after group, edge order): 16-bit fields, groups
                // 0, 1 and 2, 3
                const unsigned cnt = byte_popc(W0) + byte_popc(W1);
                const unsigned cl = __byte_perm(cnt, 0u, 0x4140), ch = __byte_perm(cnt, 0u, 0x4342);
                const unsigned il = lane_scan(cl), ih = lane_scan(ch);
                const unsigned tl = __shfl_sync(FULLMASK, il, 31), th = __shfl_sync(FULLMASK, ih, 31);
                const unsigned o1 = tl & 0xffffu, o2 = o1 + (tl >> 16), o3 = o2 + (th & 0xffffu);
                const int total = (int)(o3 + (th >> 16));
                const unsigned xl = il - cl, xh = ih - ch;
                // position in the run of eight edges
                const unsigned ql0 = xl - __shfl_sync(FULLMASK, xl, lane & ~3);
                const unsigned qh0 = xh - __shfl_sync(FULLMASK, xh, lane & ~3);
                for (int cb = 0; cb < total; cb += 32) {
                    unsigned pl = xl + (o1 << 16), ph = xh + (o2 | o3 << 16), ql = ql0, qh = qh0;
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        unsigned x = h ? W1 : W0;
                        while (x) {
                            int q = __ffs(x) - 1;
                            x &= x - 1u;
                            int sh = (q & 8) << 1;
                            unsigned one = 1u << sh, p, ol;
                            if (q < 16) {
                                p = (pl >> sh) & 0xffffu; ol = (ql >> sh) & 7u;
                                pl += one; ql += one;
                            } else {
                                p = (ph >> sh) & 0xffffu; ol = (qh >> sh) & 7u;
                                ph += one; qh += one;
                            }
                            p -= (unsigned)cb;
                            if (p < 32u)
                                list[p] = (unsigned)q | (unsigned)(2 * lane + h) << 5 | ol << 11;
                        }
                    }
                    __syncwarp();
                    const bool has = cb + lane < total;
                    const unsigned code = has ? list[lane] : 0u;
                    const int kk = (int)((code >> 3) & 3u);
                    const int jk = of(j, kk), nuk = of(nu, kk), boxk = of(box, kk), e0k = of(e0, kk);
                    const Real uk = of(u, kk), sk = of(sig_nhi, kk);
                    int bin = -1;
                    if (has)
                        bin = gas_contribution<Real, G, BAR, SH>(P, (long long)e0k + eb + ((code >> 5) & 63u),
                                                                 code & 7u, jk, nuk, boxk, uk, sk, sv, lane);
                    merge(kk, bin, (int)(code >> 11));
                }
            }
            // the staged contributions, group after group
            const int f1 = of(fc, 0), f2 = f1 + of(fc, 1), f3 = f2 + of(fc, 2), ft = f3 + of(fc, 3);
            for (int cb = 0; cb < ft; cb += 32) {
                const int p = cb + lane;
                const int kk = (p >= f1) + (p >= f2) + (p >= f3);
                const int c = p - (kk == 0 ? 0 : kk == 1 ? f1 : kk == 2 ? f2 : f3);
                const int sok = of(so, kk), nuk = of(nu, kk);
                int bin = -1;
                if (p < ft) bin = staged_contribution<Real, SH>(P, fcur, P.seg_ent[sok + c], nuk, sv, lane);
                merge(kk, bin, c & 7);
            }
            // the merged packets
            const Real N = a.photons();
            const bool occ = kv && N > Real(0);
            const bool act = occ && (a.clock() / N < (Real)P.dt);
            const unsigned bo = (__ballot_sync(FULLMASK, occ) >> (8 * kq)) & 0xffu;
            const unsigned ba = (__ballot_sync(FULLMASK, act) >> (8 * kq)) & 0xffu;
            if (occ) a.store(Sn, (Real *)P.slG[nxt], sidx, gidx, sgs);
            Real av = ab.A.get().x, ae = ab.A.get().y, w = ab.W.get();
#pragma unroll
            for (int o = G >> 1; o > 0; o >>= 1) {
                av += __shfl_down_sync(FULLMASK, av, o, G);
                ae += __shfl_down_sync(FULLMASK, ae, o, G);
                w += __shfl_down_sync(FULLMASK, w, o, G);
            }
            if (kv && bl == 0) {
                P.occ[nxt][key] = bo;
                P.act[nxt][key] = ba;
                atomicAdd(&stot[0], __popc(bo));
                atomicAdd(&stot[1], __popc(ba));
                if (touched || fc > 0) {
                    bad |= pend > (1ull << 62);
                    pend = deposit_group<Real>(P, key, j, box, av, ae, w);
                }
            }
        } else {
            // 32 cones: the words of up to 64 edges of each group (lane: edges 2 lane, 2 lane + 1)
            unsigned w0[4], w1[4];
            int nk[4];             // contributions of the group; 33: a warp of its own
            unsigned cnt = 0u;     // gas contributions of the lane's edges, eight bits a group
            const bool narrow = kv && park == 0u && ne <= 64;
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                int rem = of((int)narrow, kk) ? of(ne, kk) - 2 * lane : 0;
                const unsigned *bw = P.bm + (long long)of(nu, kk) * P.n * P.kn + of(e0, kk) + 2 * lane;
                w0[kk] = rem > 0 ? bw[0] : 0u;
                w1[kk] = rem > 1 ? bw[1] : 0u;
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
                int pc = __popc(w0[kk]) + __popc(w1[kk]);
                nk[kk] = __reduce_add_sync(FULLMASK, pc) + of(fc, kk);
                if (!of((int)narrow, kk) || nk[kk] > 32) {
                    nk[kk] = 33;
                    w0[kk] = w1[kk] = 0u;
                } else {
                    cnt |= (unsigned)pc << (8 * kk);
                    unsigned *bw = P.bm + (long long)of(nu, kk) * P.n * P.kn + of(e0, kk) + 2 * lane;
                    if (w0[kk]) bw[0] = 0u;
                    if (w1[kk]) bw[1] = 0u;
                }
            }
            const unsigned incl = lane_scan(cnt), excl = incl - cnt;
            const unsigned tot = __shfl_sync(FULLMASK, incl, 31);
            const unsigned mid = __shfl_sync(FULLMASK, excl, 16);   // of the first 32 edges
            const int nvalid = (int)(gb1 - g0 < 4 ? gb1 - g0 : 4);
            for (int k0 = 0; k0 < nvalid;) {
                // groups k0 .. k1 - 1 together
                int k1 = k0, n = 0, ngas = 0;
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                    if (kk == k1 && kk < nvalid && kk >= k0 && n + nk[kk] <= 32) {
                        n += nk[kk];
                        ngas += (int)((tot >> (8 * kk)) & 0xffu);
                        k1 = kk + 1;
                    }
                if (k1 == k0) {
                    wide_group<Real, BAR, SH>(P, cur, fcur, of(key, k0), of((int)touched, k0) != 0,
                                              of(fc, k0), of(so, k0), sv, list, smask[wid][0], pend,
                                              bad, stot);
                    ++k0;
                    continue;
                }
                smask[wid][0][lane] = 0u;
                smask[wid][1][lane] = 0u;
                // the list: gas contributions group after group (in edge order), then staged
                // ones; gk, sk, vk: the lane's group's first gas and staged entries, and its
                // first lane of the absorption sums
                int goff = 0, soff = ngas, voff = 0;
                int myk = -1, gk = 0, m0 = 0, m1 = 0, sk = 0, m2 = 0, vk = 0;   // absorption sums
                int ek = k0, ec = 0;                                             // staged entry
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    if (kk < k0 || kk >= k1) continue;
                    int gas = (int)((tot >> (8 * kk)) & 0xffu), half = (int)((mid >> (8 * kk)) & 0xffu);
                    int st = of(fc, kk);
                    int M = max(max(half, gas - half), st);
                    if (lane >= voff && lane < voff + M) {
                        myk = kk; gk = goff; m0 = half; m1 = gas - half; sk = soff; m2 = st; vk = voff;
                    }
                    if (lane >= soff && lane < soff + st) { ek = kk; ec = lane - soff; }
                    int p = goff + (int)((excl >> (8 * kk)) & 0xffu);
                    for (unsigned x = w0[kk]; x; x &= x - 1u)
                        list[p++] = (unsigned)(__ffs(x) - 1) | (unsigned)(2 * lane) << 5 | (unsigned)kk << 11;
                    for (unsigned x = w1[kk]; x; x &= x - 1u)
                        list[p++] = (unsigned)(__ffs(x) - 1) | (unsigned)(2 * lane + 1) << 5 | (unsigned)kk << 11;
                    goff += gas;
                    soff += st;
                    voff += M;
                }
                __syncwarp();
                const bool gas = lane < ngas;
                const unsigned code = gas ? list[lane] : 0u;
                const int kk = gas ? (int)(code >> 11) : ek;
                const int jk = of(j, kk), nuk = of(nu, kk), boxk = of(box, kk), e0k = of(e0, kk),
                          sok = of(so, kk);
                const Real uk = of(u, kk), snk = of(sig_nhi, kk);
                int bin = -1;
                if (gas)
                    bin = gas_contribution<Real, G, BAR, SH>(P, (long long)e0k + ((code >> 5) & 63u),
                                                             code & 31u, jk, nuk, boxk, uk, snk, sv, lane);
                else if (lane < n)
                    bin = staged_contribution<Real, SH>(P, fcur, P.seg_ent[sok + ec], nuk, sv, lane);
                __syncwarp();
                // the lowest lane of each (group, cone) adds its contributions in list order
                const unsigned live = __ballot_sync(FULLMASK, bin >= 0);
                unsigned peers = __match_any_sync(FULLMASK, bin >= 0 ? 32 * kk + bin : 128 + lane);
                if (bin >= 0 && (peers & ((1u << lane) - 1u)) == 0u) {
                    const bool sgs = SH && nuk == 0;
                    ConeSum<Real, SH> a;
                    a.zero();
                    do {
                        int t = __ffs(peers) - 1;
                        peers &= peers - 1u;
                        a.add(sv, t, sgs);
                    } while (peers);
                    const Real N = a.photons();
                    if (N > Real(0)) {
                        a.store(Sn, (Real *)P.slG[nxt], (long long)jk * P.S + (long long)nuk * G + bin,
                                (long long)jk * G + bin, sgs);
                        atomicOr(&smask[wid][0][kk], 1u << bin);
                        if (a.clock() / N < (Real)P.dt) atomicOr(&smask[wid][1][kk], 1u << bin);
                    }
                }
                // absorption sums: lane i of a group's adds the i-th contributions of its two
                // runs of 32 edges and of its staged ones, then a tree over the lanes
                AbsSum<Real> ab;
                ab.zero();
                const int i = lane - vk;
                auto take = [&](bool on, int t) {
                    if (on && ((live >> t) & 1u)) ab.add(sv, t);
                };
                if (myk >= 0) {
                    take(i < m0, (gk + i) & 31);
                    take(i < m1, (gk + m0 + i) & 31);
                    take(i < m2, (sk + i) & 31);
                }
                const int M = myk >= 0 ? max(max(m0, m1), m2) : 0;
                Real av = ab.A.get().x, ae = ab.A.get().y, w = ab.W.get();
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) {
                    Real v0 = __shfl_down_sync(FULLMASK, av, o), v1 = __shfl_down_sync(FULLMASK, ae, o),
                         v2 = __shfl_down_sync(FULLMASK, w, o);
                    if (i + o < M) { av += v0; ae += v1; w += v2; }
                }
                __syncwarp();
                if ((lane & 7) == 0 && kq >= k0 && kq < k1) {
                    const unsigned bo = smask[wid][0][kq], ba = smask[wid][1][kq];
                    P.occ[nxt][key] = bo;
                    P.act[nxt][key] = ba;
                    atomicAdd(&stot[0], __popc(bo));
                    atomicAdd(&stot[1], __popc(ba));
                }
                const long long keyk = of(key, myk >= 0 ? myk : 0);
                const int jd = of(j, myk >= 0 ? myk : 0), boxd = of(box, myk >= 0 ? myk : 0);
                if (myk >= 0 && i == 0) {
                    bad |= pend > (1ull << 62);
                    pend = deposit_group<Real>(P, keyk, jd, boxd, av, ae, w);
                }
                __syncwarp();
                k0 = k1;
            }
        }
    }
    bad |= pend > (1ull << 62);
    if (bad) atomicOr((unsigned long long *)&P.cnt[CNT_ERR], (unsigned long long)ERRB_RANGE);
    __syncthreads();
    if (threadIdx.x == 0 && stot[0]) {
        atomicAdd((unsigned long long *)&P.cnt[CNT_OUT], (unsigned long long)stot[0]);
        atomicAdd((unsigned long long *)&P.cnt[CNT_ACTIVE], (unsigned long long)stot[1]);
        atomicAdd((unsigned long long *)&P.cnt[CNT_ACTS], (unsigned long long)stot[1]);
    }
}

// bookkeeping of the hop loop (single thread)
enum { HL_END = 2, HL_TRANSPORT = 4, HL_STEP = 5 };
// in_graph: the launch is a node of the step graph; `loop` is the hop loop's conditional and
// `pair` the switch that picks the copy of the next hop (its slot and free-packet buffers)
__global__ void k_hop_lens(DevPtrs P, int *lens, int phase, long long arg, int in_graph,
                           cudaGraphConditionalHandle loop, cudaGraphConditionalHandle pair) {
    long long *cnt = P.cnt;
    if (phase == HL_STEP) {             // the step number (arg)
        cnt[CNT_STEP] = arg;
        return;
    }
    if (phase == HL_END) {              // after the hop (arg = hop cap)
        long long nr = lens[2];
        if (nr > P.F_cap) cnt[CNT_ERR] |= ERRB_FREE_CAP;
        if (lens[3] > P.ST_cap) cnt[CNT_ERR] |= ERRB_STAGE_CAP;
        cnt[CNT_NREQ] = nr;
        lens[0] = (int)(nr < P.F_cap ? nr : P.F_cap);
        cnt[CNT_VIRT] += lens[0];
        cnt[CNT_STG] += lens[3];
        cnt[CNT_WLS] += lens[4];
        if (nr > cnt[CNT_PKFREE]) cnt[CNT_PKFREE] = nr;
        if (cnt[CNT_ACTIVE] > cnt[CNT_PKACT]) cnt[CNT_PKACT] = cnt[CNT_ACTIVE];
        cnt[CNT_CUR] ^= 1;              // the receivers' buffers hold the next hop's packets
        cnt[CNT_FCUR] ^= 1;
        long long hop = ++cnt[CNT_HOP];
        // another hop while packets still move and no error stopped the step; at the hop cap
        // the free packets in flight are dropped (counted escaped) and the step reports it
        bool moving = cnt[CNT_ACTIVE] != 0 || cnt[CNT_LIVE] != 0;
        bool more = moving && cnt[CNT_ERR] == 0;
        if (more && hop >= arg) {
            more = false;
            cnt[CNT_DROP] = 1;
        }
        cnt[CNT_MORE] = more ? 1 : 0;
        if (in_graph) cudaGraphSetConditional(loop, more ? 1u : 0u);
    } else {                            // HL_TRANSPORT: start of the hop loop (arg = hop cap)
        cnt[CNT_VIRT] = 0;
        cnt[CNT_VESC] = 0;
        for (int k = CNT_ACTP; k <= CNT_OUT; ++k) cnt[k] = 0;
        cnt[CNT_HOP] = 0;
        cnt[CNT_PKFREE] = 0;
        cnt[CNT_PKACT] = 0;
        cnt[CNT_DROP] = arg <= 0 ? 1 : 0;
    }
    // counters of the next hop
    cnt[CNT_ACTIVE] = 0;
    cnt[CNT_LIVE] = 0;
    cnt[CNT_VQ] = 0;                    // the virtual particles' work queue
    lens[2] = lens[3] = lens[4] = lens[5] = 0;
    // in the graph: which of the four copies of the hop (slot and free-packet buffers) runs next
    if (in_graph) cudaGraphSetConditional(pair, (unsigned)(cnt[CNT_CUR] | (cnt[CNT_FCUR] << 1)));
}

// The hop loop stopped with packets still moving (hop cap, or an error): the particles that
// would have sent next are counted like every hop's.  At the hop cap the free packets in flight
// leave the box (counted escaped).  Does nothing after a loop that ran out of packets.
template <typename Real>
__global__ void k_drop_free(DevPtrs P, const int *lens) {
    if (!P.cnt[CNT_DROP] && !P.cnt[CNT_ERR]) return;
    const long long t0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const long long stride = (long long)gridDim.x * blockDim.x;
    const unsigned *act = P.act[(int)P.cnt[CNT_CUR]];
    for (long long i = t0; i < P.n; i += stride) {
        unsigned any = 0u;
        for (int nu = 0; nu < P.nf; ++nu) any |= act[i * P.nf + nu];
        if (any) atomicAdd((unsigned long long *)&P.cnt[CNT_ACTP], 1ull);
    }
    if (!P.cnt[CNT_DROP]) return;
    FreeBuf F = P.fr[(int)P.cnt[CNT_FCUR]];
    for (long long f = t0; f < lens[0]; f += stride) {
        Real N = ((Real *)F.N)[f];
        if (N > Real(0)) {
            int b = F.box[f];
            atomicAdd(&P.esc_fx[b], esc_fixed(N, P, b));
            ((Real *)F.N)[f] = Real(0);
        }
    }
}

// ------------------------------------------------------------------------------------------
// host orchestration
// ------------------------------------------------------------------------------------------

#define LAUNCH_ON(sx, id, n, ...)   \
    do {                            \
        kt_begin(c, id, sx);        \
        __VA_ARGS__;                \
        kt_end(c, id, sx, n);       \
    } while (0)
#define LAUNCH(id, n, ...) LAUNCH_ON(st, id, n, __VA_ARGS__)

// the step number the rotations and virtual particles draw with (kept on the device)
static void set_step(rt_ctx *c, long long step, cudaStream_t st) {
    if (c->step_dev == step && step != LLONG_MIN) return;
    LAUNCH(KT_HOP_LENS, 1, (k_hop_lens<<<1, 1, 0, st>>>(c->d, c->hop.lens, HL_STEP, step, 0, 0, 0)));
    c->step_dev = step;
}

// Particles a warp of the sender side takes together: as many as its 32 (particle, frequency)
// words hold, but no more than leave the resident warps a turn each, since a small box needs its
// particles spread over the chip more than it needs full lanes: 32 warps an SM with FP32
// packets; 8 with FP64 packets, where a few warps already fill the FP64 pipe and fuller lanes
// mean fewer of its instructions (the 16^3 sphere's step: 1.79 ms with 32, 1.67 with 8, 1.73 with 4).
// nu0: the launch's first frequency.
static int send_turn(const DevPtrs &P, int nu0) {
    long long most = std::max(1, 32 / (P.nf - nu0));
    return (int)std::min(most, std::max(1ll, P.n / (152 * (P.fp32 ? 32 : 8))));
}

// The sender side of a hop (lens: its counts; null: inspection, no requests), 32 frequencies a launch.
template <typename Real, int NRC>
static void launch_senders(rt_ctx *c, cudaStream_t st, int cur, int max_blocks, int *lens) {
    const DevPtrs &P = c->d;
    const int tb = 256;
    for (int nu0 = 0; nu0 < P.nf; nu0 += 32) {
        const int per = send_turn(P, nu0), nfl = std::min(32, P.nf - nu0);
        const int nb = rt_blocks((P.n + per - 1) / per * 32, tb, max_blocks);
        auto kernel = P.nf <= 32 ? (P.shared ? k_phaseA<Real, NRC, true, false> : k_phaseA<Real, NRC, false, false>)
                                 : (P.shared ? k_phaseA<Real, NRC, true, true> : k_phaseA<Real, NRC, false, true>);
        LAUNCH(KT_PHASE_A, 1, (kernel<<<nb, tb, 0, st>>>(P, cur, per, nu0, nfl, lens)));
    }
}

// One hop, in six launches and a bookkeeping kernel (k_hop_lens HL_END, launched by the
// caller), with no pass over a capacity.  Two streams:
//   st: gas senders; virtual particles (after both senders)
//   s2: free-packet senders; work list (after both senders); segments; receiver side
// The caller's stream continues after the receiver side.  What a small box costs is its
// chain of dependent launches: 5 here (senders, work list, segments, receiver side,
// bookkeeping), where the hop was 20 launches with a chain of 15 before: the 12^3 sphere's step
// of 10 hops went from 0.90 to 0.50 ms, that of a 64^3 box with hardly any packets and 39 hops
// from 6.1 to 3.4 ms.
// nfr bounds the free packets of the hop (their count is on the device); cur and fcur are the
// hop's slot and free-packet buffers.
template <typename Real, int NRC>
static void hop_core(rt_ctx *c, cudaStream_t st, long long nfr, int cur, int fcur) {
    DevPtrs &P = c->d;
    const int GA = c->grid_hop[0] ? c->grid_hop[0] : GRID_A;
    const int GV = c->grid_hop[1] ? c->grid_hop[1] : GRID_V;
    const int GB = c->grid_hop[2] ? c->grid_hop[2] : GRID_B;
    HopScratch &H = c->hop;
    const int tb = 256;
    long long nkey = P.n * P.nf;
    cudaStream_t s2 = c->st2;
    cudaEvent_t evFork = c->hev[0], evA = c->hev[1], evFree = c->hev[2], evB = c->hev[3];
    if (nfr < 1) nfr = 1;
    cudaEventRecord(evFork, st);
    cudaStreamWaitEvent(s2, evFork, 0);
    // instances: the common case; with a barrier; with a shared frequency bin (whose instance
    // also takes the barrier test, which is a no-op in boxes without one)
    const int nbf = rt_blocks(nfr * 32, tb, GRID_F);
    if (P.shared)
        LAUNCH_ON(s2, KT_FREE_A, 1, (k_free<Real, NRC, true, true><<<nbf, tb, 0, s2>>>(P, fcur, H.lens)));
    else if (P.any_bar)
        LAUNCH_ON(s2, KT_FREE_A, 1, (k_free<Real, NRC, true, false><<<nbf, tb, 0, s2>>>(P, fcur, H.lens)));
    else
        LAUNCH_ON(s2, KT_FREE_A, 1, (k_free<Real, NRC, false, false><<<nbf, tb, 0, s2>>>(P, fcur, H.lens)));
    cudaEventRecord(evFree, s2);
    launch_senders<Real, NRC>(c, st, cur, GA, H.lens);
    cudaEventRecord(evA, st);
    cudaStreamWaitEvent(s2, evA, 0);
    LAUNCH_ON(s2, KT_WORKLIST, 1, (k_worklist<<<rt_blocks(nkey, 1024, 152 * 8), tb, 0, s2>>>(P, cur, H.lens)));
    LAUNCH_ON(s2, KT_SEG_FILL, 1, (k_seg_fill<<<rt_blocks(nfr * 2, tb, 152 * 8), tb, 0, s2>>>(P, fcur, H.lens)));
    cudaStreamWaitEvent(st, evFree, 0);
    const int nbb = rt_blocks(nkey * 8, tb, GB);
    if (P.shared)
        LAUNCH_ON(s2, KT_PHASE_B, 1, (k_phaseB<Real, NRC, true, true><<<nbb, tb, 0, s2>>>(P, cur, fcur, H.lens)));
    else if (P.any_bar)
        LAUNCH_ON(s2, KT_PHASE_B, 1, (k_phaseB<Real, NRC, true, false><<<nbb, tb, 0, s2>>>(P, cur, fcur, H.lens)));
    else
        LAUNCH_ON(s2, KT_PHASE_B, 1, (k_phaseB<Real, NRC, false, false><<<nbb, tb, 0, s2>>>(P, cur, fcur, H.lens)));
    cudaEventRecord(evB, s2);
    const int IS = KNN_IB_SMALL, IL = KNN_IB_LARGE;
    const int nbv = rt_blocks(P.F_cap * 32, tb, GV);
    if (P.kwide && P.shared)   // boxes above 2^22 particles: the general instance, 24-bit keys
        LAUNCH(KT_VIRTUAL, 1, (k_virtual<Real, NRC, true, true, IL><<<nbv, tb, 0, st>>>(P, cur, fcur, H.lens)));
    else if (P.kwide)
        LAUNCH(KT_VIRTUAL, 1, (k_virtual<Real, NRC, true, false, IL><<<nbv, tb, 0, st>>>(P, cur, fcur, H.lens)));
    else if (P.shared)
        LAUNCH(KT_VIRTUAL, 1, (k_virtual<Real, NRC, true, true, IS><<<nbv, tb, 0, st>>>(P, cur, fcur, H.lens)));
    else if (P.any_bar)
        LAUNCH(KT_VIRTUAL, 1, (k_virtual<Real, NRC, true, false, IS><<<nbv, tb, 0, st>>>(P, cur, fcur, H.lens)));
    else
        LAUNCH(KT_VIRTUAL, 1, (k_virtual<Real, NRC, false, false, IS><<<nbv, tb, 0, st>>>(P, cur, fcur, H.lens)));
    cudaStreamWaitEvent(st, evB, 0);
}

static void graph_destroy(rt_ctx *c);
void rt_launch_grids(const rt_ctx *c, long long out[3]) {
    const int def[3] = {GRID_A, GRID_V, GRID_B};
    for (int k = 0; k < 3; ++k) out[k] = c->grid_hop[k] ? c->grid_hop[k] : def[k];
}

// cone bitmaps and receiver flags back to zero (as every hop leaves them)
static void clear_cone_bits(rt_ctx *c, cudaStream_t st) {
    DevPtrs &P = c->d;
    cudaMemsetAsync(P.bm, 0, sizeof(unsigned) * P.n * P.kn * P.nf, st);
    cudaMemsetAsync(P.touched, 0, P.n * P.nf, st);
}

// start of the hop loop: cone bits cleared if an inspection pass left some, counters reset
static void transport_begin(rt_ctx *c, cudaStream_t st) {
    DevPtrs &P = c->d;
    if (c->bm_dirty) {
        clear_cone_bits(c, st);
        c->bm_dirty = false;
    }
    LAUNCH(KT_HOP_LENS, 1, (k_hop_lens<<<1, 1, 0, st>>>(P, c->hop.lens, HL_TRANSPORT, c->cfg.hop_cap, 0, 0, 0)));
}

// after the hop loop (the counters are in cnt_h): statistics, modelled bytes, status
static rt_status transport_end(rt_ctx *c, bool fp32) {
    DevPtrs &P = c->d;
    long long hops = c->cnt_h[CNT_HOP];
    // the active packets of the first hop were made by the emission: add them to the model
    // counts below (CNT_ACTS/ACTP count those produced by each hop's receiver side)
    {
        const double R = fp32 ? 4.0 : 8.0, kn = P.kn;
        double actp = (double)c->cnt_h[CNT_ACTP], acts = (double)c->cnt_h[CNT_ACTS];
        double gcon = (double)c->cnt_h[CNT_GCON], stg = (double)c->cnt_h[CNT_STG];
        double wls = (double)c->cnt_h[CNT_WLS], outs = (double)c->cnt_h[CNT_OUT];
        double vreq = (double)c->cnt_h[CNT_VIRT];
        // algorithmic bytes: each input read once and each output written once
        const double keys = (double)hops * (double)P.n * P.nf;   // words swept over the hops
        c->kstat[KT_PHASE_A].bytes += keys * 4 + actp * kn * 20 + acts * 12 * R + gcon * 5;
        c->kstat[KT_WORKLIST].bytes += keys * 21 + wls * 4;
        c->kstat[KT_PHASE_B].bytes += wls * (16 + 8 + 48 + kn * 4) + gcon * (16 + 6 * R + 4) +
                                      stg * (12 + 8 * R) + outs * 6 * R;
        c->kstat[KT_VIRTUAL].bytes += vreq * (8 + 6 * R + 40 + kn * (16 + 4 * R + 16 + 4) +
                                              6 * R + 40);
    }
    c->stats[0] = hops;
    c->stats[1] = c->cnt_h[CNT_VIRT];
    c->stats[2] = c->cnt_h[CNT_VESC];
    c->stats[5] = c->cnt_h[CNT_PKFREE];
    c->stats[6] = c->cnt_h[CNT_PKACT];
    c->stats[7] = c->cnt_h[CNT_GCON];
    c->stats[8] = c->cnt_h[CNT_ACTP];
    c->stats[9] = c->cnt_h[CNT_ACTS];
    c->stats[10] = c->cnt_h[CNT_STG];
    c->stats[11] = c->cnt_h[CNT_WLS];
    c->stats[12] = c->cnt_h[CNT_OUT];
    long long e = c->cnt_h[CNT_ERR];
    if (e & ERRB_FREE_CAP) return rt_fail(c, RT_ERR_CAPACITY, "free packets exceeded free_cap");
    if (e & ERRB_STAGE_CAP) return rt_fail(c, RT_ERR_CAPACITY, "staged contributions exceeded capacity");
    if (e & ERRB_RANGE) return rt_fail(c, RT_ERR_RANGE, "virtual deposit overflowed its accumulator");
    if (e & ERRB_KNN)
        return rt_fail(c, RT_ERR_KNN, "a virtual particle's n_ngb-th neighbour lies beyond the kNN key range");
    if (c->cnt_h[CNT_DROP]) return rt_fail(c, RT_ERR_HOP_LIMIT, "hop loop reached hop_cap");
    return RT_OK;
}

template <typename Real> static void clear_deposits(rt_ctx *c, cudaStream_t st) {
    LAUNCH(KT_EMIT_REC, 1, (k_clear_deposits<Real><<<rt_blocks(c->d.n * c->d.nf, 256, 152 * 16), 256, 0, st>>>(c->d)));
}

template <typename Real, int NRC>
static rt_status run_parts(rt_ctx *c, int part, long long step, cudaStream_t st) {
    DevPtrs &P = c->d;
    const int tb = 256;
    long long n = P.n;
    long long nkey = n * P.nf;
    HopScratch &H = c->hop;
    if (part == 0) {  // rotations
        if (!c->capturing) set_step(c, step, st);
        long long t = n + (long long)P.ns * P.K;
        LAUNCH(KT_ROTATE, 1, (k_rotate<<<(unsigned)((t + tb - 1) / tb), tb, 0, st>>>(P)));
        return rt_cuda_check(c, cudaGetLastError(), "rotate");
    }
    if (part == 1) {  // re-bin held packets
        LAUNCH(KT_REBIN, 1, (k_rebin<Real, NRC><<<(unsigned)((nkey + tb - 1) / tb), tb, 0, st>>>(P)));
        return rt_cuda_check(c, cudaGetLastError(), "rebin");
    }
    if (part == 2) {  // emission
        long long np_s = (long long)P.ns * P.K * P.nfs * P.nec;
        long long np_r = P.rec_mode == RT_REC_EMISSION_CONES ? n * P.K * P.nec : 0;
        long long np = np_s + np_r;
        if (np > P.F_cap) return rt_fail(c, RT_ERR_CAPACITY, "source packets exceed free_cap");
        if (!c->capturing) set_step(c, step, st);
        if (!c->capturing) clear_deposits<Real>(c, st);   // (the step graph has it on its other branch)
        LAUNCH(KT_EMIT_REC, 1, (k_emit_rec<Real, NRC><<<(unsigned)((n + tb - 1) / tb), tb, 0, st>>>(P, H.lens, (int)np)));
        c->fcur = 0;
        if (np_s > 0)
            LAUNCH(KT_EMIT_SRC, 1, (k_emit_src<Real><<<(unsigned)((np_s + tb - 1) / tb), tb, 0, st>>>(P)));
        if (np_r > 0)
            LAUNCH(KT_EMIT_SRC, 1, (k_emit_rec_cones<Real><<<(unsigned)((np_r + tb - 1) / tb), tb, 0, st>>>(P, np_s)));
        c->nfree_h = np;
        return rt_cuda_check(c, cudaGetLastError(), "emit");
    }
    if (part == 3) {  // cone masks of the held packets only (inspection)
        clear_cone_bits(c, st);
        c->bm_dirty = true;
        launch_senders<Real, NRC>(c, st, c->cur, 152 * 64, nullptr);
        return rt_cuda_check(c, cudaGetLastError(), "cone masks");
    }
    // part 4: the hop loop, driven from the host (one synchronisation per hop)
    set_step(c, step, st);
    transport_begin(c, st);
    for (;;) {
        hop_core<Real, NRC>(c, st, c->nfree_h, c->cur, c->fcur);
        LAUNCH(KT_HOP_LENS, 1, (k_hop_lens<<<1, 1, 0, st>>>(P, H.lens, HL_END, c->cfg.hop_cap, 0, 0, 0)));
        c->cur ^= 1;
        c->fcur ^= 1;
        cudaMemcpyAsync(c->cnt_h, P.cnt, sizeof(long long) * CNT_N, cudaMemcpyDeviceToHost, st);
        rt_status hs = rt_cuda_check(c, cudaStreamSynchronize(st), "hop");
        if (hs != RT_OK) return hs;
        kt_resolve(c);
        c->nfree_h = std::min<long long>(c->cnt_h[CNT_NREQ], P.F_cap);
        if (c->cnt_h[CNT_MORE]) continue;
        if (c->cnt_h[CNT_ERR] || c->cnt_h[CNT_DROP])
            LAUNCH(KT_DROP, 1, (k_drop_free<Real><<<rt_blocks(std::max(P.F_cap, n), tb, 152 * 64), tb, 0, st>>>(P, H.lens)));
        break;
    }
    cudaMemcpyAsync(c->cnt_h, P.cnt, sizeof(long long) * CNT_N, cudaMemcpyDeviceToHost, st);
    rt_status hs = rt_cuda_check(c, cudaStreamSynchronize(st), "hop loop");
    if (hs != RT_OK) return hs;
    kt_resolve(c);
    return transport_end(c, sizeof(Real) == 4);
}

// ---- the whole step as one CUDA graph --------------------------------------------------
// Prologue (rotations, re-binning, emission, emitted-photon tally, counter reset), a
// conditional while node whose body is one hop (its last kernel decides whether another hop
// runs), and the epilogue (drop at the hop cap, chemistry, end-of-step tally).  Captured on
// the context's own streams.  What changes from step to step or hop to hop is on the device:
// the step and hop numbers (read where they are used), and the buffer pair of the hop, which
// selects one of four captured copies of the hop through a switch node, so that inside a
// copy the buffers are launch parameters.  One capture serves every step.
static void graph_destroy(rt_ctx *c) {
    if (c->graph_exec) cudaGraphExecDestroy(c->graph_exec);
    if (c->graph) cudaGraphDestroy(c->graph);
    c->graph_exec = nullptr;
    c->graph = nullptr;
}

static rt_status capture_segment(rt_ctx *c, cudaGraph_t *out, rt_status (*body)(rt_ctx *, cudaStream_t)) {
    cudaStream_t sc = c->st_cap;
    cudaError_t e = cudaStreamBeginCapture(sc, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return rt_cuda_check(c, e, "graph capture");
    rt_status s = body(c, sc);
    cudaGraph_t g = nullptr;
    cudaError_t e2 = cudaStreamEndCapture(sc, &g);
    if (s != RT_OK) {
        if (g) cudaGraphDestroy(g);
        return s;
    }
    if (e2 != cudaSuccess) return rt_cuda_check(c, e2, "graph capture");
    *out = g;
    return RT_OK;
}

template <typename Real, int NRC>
static rt_status seg_prologue(rt_ctx *c, cudaStream_t st) {
    rt_status s;
    // beside the rest: the deposit words cleared, and the emitted-photon tally (it reads what the
    // last step's chemistry left)
    cudaEventRecord(c->hev[0], st);
    cudaStreamWaitEvent(c->st2, c->hev[0], 0);
    clear_deposits<Real>(c, c->st2);
    if ((s = rt_budget_launch(c, 0, c->st2))) return s;
    cudaEventRecord(c->hev[1], c->st2);
    if ((s = run_parts<Real, NRC>(c, 0, 0, st))) return s;
    if ((s = run_parts<Real, NRC>(c, 1, 0, st))) return s;
    if ((s = run_parts<Real, NRC>(c, 2, 0, st))) return s;
    LAUNCH(KT_HOP_LENS, 1, (k_hop_lens<<<1, 1, 0, st>>>(c->d, c->hop.lens, HL_TRANSPORT, c->cfg.hop_cap, 1, c->loop_h, c->pair_h)));
    cudaStreamWaitEvent(st, c->hev[1], 0);
    return rt_cuda_check(c, cudaGetLastError(), "graph prologue");
}

template <typename Real>
static rt_status seg_epilogue(rt_ctx *c, cudaStream_t st) {
    LAUNCH(KT_DROP, 1, (k_drop_free<Real><<<rt_blocks(std::max(c->d.F_cap, c->d.n), 256, 152 * 8), 256, 0, st>>>(c->d, c->hop.lens)));
    rt_status s;
    if ((s = rt_chem_launch(c, st))) return s;
    if ((s = rt_budget_launch(c, 1, st))) return s;
    return rt_cuda_check(c, cudaGetLastError(), "graph epilogue");
}

// The while node's body: a switch node over the four (slot buffer, free-packet buffer) pairs,
// each body one capture of the hop with those buffers as launch parameters, then HL_END (sets
// the loop condition, and the switch for the next hop; the first hop's was set before the loop).
template <typename Real, int NRC>
static cudaError_t build_hop_body(rt_ctx *c, cudaGraph_t body) {
    cudaGraphNode_t nsw, nend;
    cudaGraphNodeParams cp = {};
    cp.type = cudaGraphNodeTypeConditional;
    cp.conditional.handle = c->pair_h;
    cp.conditional.type = cudaGraphCondTypeSwitch;
    cp.conditional.size = 4;
    cudaError_t e = cudaGraphAddNode(&nsw, body, nullptr, nullptr, 0, &cp);
    c->in_hop_body = true;
    long long once[KT_N];
    for (int par = 0; par < 4 && e == cudaSuccess; ++par) {
        e = cudaStreamBeginCaptureToGraph(c->st_cap, cp.conditional.phGraph_out[par], nullptr,
                                          nullptr, 0, cudaStreamCaptureModeThreadLocal);
        if (e != cudaSuccess) break;
        hop_core<Real, NRC>(c, c->st_cap, c->d.F_cap, par & 1, par >> 1);
        cudaGraph_t b = cp.conditional.phGraph_out[par];
        e = cudaStreamEndCapture(c->st_cap, &b);
        // one copy runs per hop: its launches are counted once
        if (par == 0) memcpy(once, c->graph_launch_hop, sizeof(once));
        else memcpy(c->graph_launch_hop, once, sizeof(once));
    }
    if (e == cudaSuccess) {
        DevPtrs P = c->d;
        int *lens = c->hop.lens;
        int phase = HL_END, in_graph = 1;
        long long arg = c->cfg.hop_cap;
        cudaGraphConditionalHandle loop = c->loop_h, pair = c->pair_h;
        void *args[] = {&P, &lens, &phase, &arg, &in_graph, &loop, &pair};
        cudaKernelNodeParams kp = {};
        kp.func = (void *)k_hop_lens;
        kp.gridDim = dim3(1);
        kp.blockDim = dim3(1);
        kp.kernelParams = args;
        c->graph_launch_hop[KT_HOP_LENS] += 1;
        e = cudaGraphAddKernelNode(&nend, body, &nsw, 1, &kp);
    }
    c->in_hop_body = false;
    return e;
}

template <typename Real, int NRC>
static rt_status capture_step(rt_ctx *c) {
    graph_destroy(c);
    for (int k = 0; k < KT_N; ++k) c->graph_launch_step[k] = c->graph_launch_hop[k] = 0;
    c->capturing = true;
    cudaGraph_t pro = nullptr, epi = nullptr, g = nullptr;
    // the handles of the hop loop and of its switch, set by kernels of the prologue and the body
    cudaError_t e = cudaGraphCreate(&g, 0);
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&c->loop_h, g, 1, cudaGraphCondAssignDefault);
    if (e == cudaSuccess) e = cudaGraphConditionalHandleCreate(&c->pair_h, g, 0, 0);
    rt_status s = rt_cuda_check(c, e, "graph build");
    if (s == RT_OK) s = capture_segment(c, &pro, seg_prologue<Real, NRC>);
    if (s == RT_OK) s = capture_segment(c, &epi, seg_epilogue<Real>);
    if (s == RT_OK) {
        cudaGraphNode_t npro, nloop, nepi;
        e = cudaGraphAddChildGraphNode(&npro, g, nullptr, 0, pro);
        cudaGraphNodeParams cp = {};
        if (e == cudaSuccess) {
            cp.type = cudaGraphNodeTypeConditional;
            cp.conditional.handle = c->loop_h;
            cp.conditional.type = cudaGraphCondTypeWhile;
            cp.conditional.size = 1;
            e = cudaGraphAddNode(&nloop, g, &npro, nullptr, 1, &cp);
        }
        if (e == cudaSuccess) e = build_hop_body<Real, NRC>(c, cp.conditional.phGraph_out[0]);
        if (e == cudaSuccess) e = cudaGraphAddChildGraphNode(&nepi, g, &nloop, 1, epi);
        if (e == cudaSuccess) e = cudaGraphInstantiate(&c->graph_exec, g, 0);
    }
    c->capturing = false;
    c->in_hop_body = false;
    if (pro) cudaGraphDestroy(pro);
    if (epi) cudaGraphDestroy(epi);
    if (s != RT_OK || e != cudaSuccess) {
        if (c->graph_exec) cudaGraphExecDestroy(c->graph_exec);
        if (g) cudaGraphDestroy(g);
        c->graph_exec = nullptr;
        cudaGetLastError();
        return s != RT_OK ? s : rt_cuda_check(c, e, "graph build");
    }
    c->graph = g;
    c->graph_P = c->d;
    c->graph_hop_cap = c->cfg.hop_cap;
    return RT_OK;
}

template <typename Real, int NRC>
static rt_status step_graph(rt_ctx *c, long long step, cudaStream_t st) {
    bool stale = !c->graph_exec || c->graph_hop_cap != c->cfg.hop_cap ||
                 memcmp(&c->graph_P, &c->d, sizeof(DevPtrs)) != 0;
    rt_status s;
    if (stale && (s = capture_step<Real, NRC>(c))) return s;
    set_step(c, step, st);
    if (c->bm_dirty) {
        clear_cone_bits(c, st);
        c->bm_dirty = false;
    }
    cudaError_t e = cudaGraphLaunch(c->graph_exec, st);
    if (e != cudaSuccess) return rt_cuda_check(c, e, "graph launch");
    cudaMemcpyAsync(c->cnt_h, c->d.cnt, sizeof(long long) * CNT_N, cudaMemcpyDeviceToHost, st);
    if ((s = rt_cuda_check(c, cudaStreamSynchronize(st), "graph step"))) return s;
    long long hops = c->cnt_h[CNT_HOP];
    for (int k = 0; k < KT_N; ++k) {
        long long l = c->graph_launch_step[k] + hops * c->graph_launch_hop[k];
        c->kstat[k].launches += l;
        c->launches += l;
    }
    c->cur = (int)c->cnt_h[CNT_CUR];
    c->fcur = (int)c->cnt_h[CNT_FCUR];
    c->nfree_h = std::min<long long>(c->cnt_h[CNT_NREQ], c->d.F_cap);
    c->stats[3] = c->cnt_h[CNT_SUB];
    c->stats[4] = c->cnt_h[CNT_FLOOR];
    rt_status ts = transport_end(c, sizeof(Real) == 4);
    return ts != RT_OK ? ts : rt_subcycle_status(c);
}

rt_status rt_step_graph(rt_ctx *c, long long step, cudaStream_t st) {
    int nrc = c->d.nrc;
    if (c->d.fp32) return nrc == 8 ? step_graph<float, 8>(c, step, st) : step_graph<float, 32>(c, step, st);
    return nrc == 8 ? step_graph<double, 8>(c, step, st) : step_graph<double, 32>(c, step, st);
}

// ---- launch-size tuning on whole steps -------------------------------------------------------
// With tune_launch the first steps run as the captured step graph, each with one triple of grid
// sizes of the sender side, the virtual particles and the receiver side, and are timed with CUDA
// events around the graph launch, so that the overlap of the two streams is in the objective.
// The time of a step is divided by its work (packets moved, particles sending, virtual
// particles: device counters of that step).  Coordinate search from the built-in sizes, the
// virtual particles first (152 x {2, 3, 4, 5} blocks: at most one wave, since its warps pull
// from a work queue; fewer blocks leave room for the receiver side beside it), then the sender
// and the receiver side (152 x {8, 16, 32, 64} blocks); each candidate step follows a step of
// the current best, so that the pair sees nearly the same work, and replaces it when it costs
// 1% less per unit of work.  The winner is kept
// for the process per (configuration, particles, boxes): a later context of the same kind
// starts with it and does not tune.  The steps run while tuning are ordinary steps: results do
// not depend on the launch sizes.
static std::mutex g_tune_mu;
static std::map<std::string, std::array<int, 3>> g_tune_cache;

static std::string tune_key(const rt_ctx *c) {
    const DevPtrs &P = c->d;
    char buf[256];
    snprintf(buf, sizeof(buf), "%lld/%d/%d/%d/%d/%d/%d/%d/%d", P.n, P.nb, P.kn, P.ntc, P.nrc,
             P.nf, P.fp32, P.rec_mode, P.shared);
    return buf;
}

static void set_grids(rt_ctx *c, const int g[3]) {
    bool same = true;
    for (int k = 0; k < 3; ++k) same &= c->grid_hop[k] == g[k];
    if (same) return;
    for (int k = 0; k < 3; ++k) c->grid_hop[k] = g[k];
    graph_destroy(c);     // the sizes are captured in the graph
}

rt_status rt_step_graph_tuned(rt_ctx *c, long long step, cudaStream_t st) {
    TuneState &U = c->tune;
    if (U.phase == 0) {   // start: a cached winner, or the candidates from the built-in sizes
        const int def[3] = {GRID_A, GRID_V, GRID_B};
        {
            std::lock_guard<std::mutex> lk(g_tune_mu);
            auto it = g_tune_cache.find(tune_key(c));
            if (it != g_tune_cache.end()) {
                set_grids(c, it->second.data());
                c->launch_tuned = true;
                return rt_step_graph(c, step, st);
            }
        }
        for (int k = 0; k < 3; ++k) U.best[k] = def[k];
        U.cand.clear();
        const int order[3] = {1, 0, 2};
        for (int kk : order)
            for (int q = 0; q < 4; ++q) {
                int g = kk == 1 ? 152 * (2 + q) : 152 * (8 << q);
                if (g != def[kk]) U.cand.push_back({kk, g});
            }
        U.phase = 1;
        U.steps = 0;
    }
    int g[3] = {U.best[0], U.best[1], U.best[2]};
    if (U.phase == 2) g[U.cand.front().first] = U.cand.front().second;
    set_grids(c, g);
    cudaEventRecord(c->tune_ev[0], st);
    rt_status s = rt_step_graph(c, step, st);
    cudaEventRecord(c->tune_ev[1], st);
    cudaError_t e = cudaEventSynchronize(c->tune_ev[1]);
    if (s != RT_OK) return s;
    float ms = 0.f;
    if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, c->tune_ev[0], c->tune_ev[1]);
    if (e != cudaSuccess) return rt_cuda_check(c, e, "launch-size tuning");
    double work = (double)(c->cnt_h[CNT_ACTS] + c->cnt_h[CNT_ACTP] + c->cnt_h[CNT_VIRT]);
    double cost = (double)ms / (work > 0.0 ? work : 1.0);
    ++U.steps;
    if (U.phase == 1) {
        U.best_cost = cost;
        U.phase = 2;
        return s;
    }
    if (cost < 0.99 * U.best_cost) {
        for (int k = 0; k < 3; ++k) U.best[k] = g[k];
    }
    U.cand.erase(U.cand.begin());
    // the next candidate of the same kernel is compared with the best found so far
    if (U.cand.empty()) {
        set_grids(c, U.best);
        c->launch_tuned = true;
        U.phase = 3;
        std::lock_guard<std::mutex> lk(g_tune_mu);
        g_tune_cache[tune_key(c)] = {U.best[0], U.best[1], U.best[2]};
    } else {
        U.phase = 1;
    }
    return s;
}

void rt_graph_destroy(rt_ctx *c) { graph_destroy(c); }

rt_status rt_run_step_parts(rt_ctx *c, int part, long long step, cudaStream_t st) {
    int nrc = c->d.nrc;
    if (c->d.fp32) {
        return nrc == 8 ? run_parts<float, 8>(c, part, step, st) : run_parts<float, 32>(c, part, step, st);
    }
    return nrc == 8 ? run_parts<double, 8>(c, part, step, st) : run_parts<double, 32>(c, part, step, st);
}
