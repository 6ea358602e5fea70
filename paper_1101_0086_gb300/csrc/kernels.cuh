// Kernels of the MPA node transform (MPA steps 2-5) and of the split-step
// comparator, on the four-step factorisation N = N1 * N2.
//
// A spectrum in natural order, k = k1 + N1 k2, is viewed as an N2 x N1
// row-major matrix.  The inverse transform is a column pass (length-N2 DFTs
// over k2, then the factor W_N^{-n2 k1}) followed by a row pass (length-N1
// DFTs over k1); row n2 then holds A(t) at t-index N2 n1 + n2 for
// n1 = 0..N1-1.  Because |A|^2 A (MPA step 4) and the split-step rotation
// are pointwise, the row pass forms them right there and starts the forward
// transform (length-N1 DFTs over n1, factor W_N^{+n2 k1}) without any
// transpose; the next column pass finishes it (length-N2 DFTs over n2) and
// leaves the spectrum in natural order again.
//
//   KC (column pass)  modes: MPA_PRE  phase exp(i beta_j) * exp(int G) -> inverse
//                             MPA_POST forward -> exp(-i beta_j) * sigma dz / exp(int G)  (V_j of Eq. (6))
//                             SS_STEP  forward -> linear step of Eq. (4) -> inverse
//                             FWD      forward only        INV  inverse only
//                             FWDF     forward, then the outer factor W_N^{+n2 k1}
//                             FWD_T, INV_T  the second pass of a transform between natural orders:
//                                      column c is the source's contiguous row c
//   KR (row pass)     modes: MPA  inverse -> 1/N -> |A|^2 A -> forward
//                             SS   inverse -> 1/N -> A exp(i s |A|^2) -> forward
//                             FWD  forward only        INV  inverse -> 1/N
//   SCAN              Eq. (6) trapezoid partial sums over the nodes for
//                     every frequency, with the phases of steps 2 and 5 where
//                     there are many, fused with step 7 on the last iteration.
#pragma once

#include <climits>
#include <type_traits>

#include "device.cuh"

namespace mpa {

enum { KC_MPA_PRE = 0, KC_MPA_POST = 1, KC_SS_STEP = 2, KC_FWD = 3, KC_INV = 4, KC_FWDF = 5, KC_FWD_T = 6, KC_INV_T = 7 };
// KR_MPA_KEEP: KR_MPA that also writes A(t) to keep (the reverse mode's
// forward recompute keeps it for the adjoint of the Kerr term)
enum { KR_MPA = 0, KR_SS = 1, KR_FWD = 2, KR_INV = 3, KR_MPA_KEEP = 4 };

// Debug build (MPA_DEBUG_BOUNDS=1): the global accesses of the MPA passes,
// the scan and the on-chip node transform are checked against the range of
// the launch's buffers (a plan's or batch's workspace, [lo, hi)); an access
// outside it sets ERR_BOUNDS in the error word and is skipped (a load reads
// zero), so a bad index is reported instead of touching memory it should
// not.  lo == nullptr (launches on caller buffers) checks nothing.  Release
// builds compile every check to true.
#ifndef MPA_DEBUG_BOUNDS
#define MPA_DEBUG_BOUNDS 0
#endif
enum { ERR_BOUNDS = 8u };
struct DbgRange {
    const char* lo;
    const char* hi;
    unsigned int* err;
};
__device__ __forceinline__ bool dbg_in(const DbgRange& d, const void* a, size_t bytes) {
    if (!d.lo) return true;
    const char* c = static_cast<const char*>(a);
    if (c >= d.lo && c + bytes <= d.hi) return true;
    atomicOr(d.err, (unsigned)ERR_BOUNDS);
    return false;
}
#if MPA_DEBUG_BOUNDS
#define MPA_DBG_OK(d, ptr, bytes) ::mpa::dbg_in((d), (ptr), (bytes))
#else
#define MPA_DBG_OK(d, ptr, bytes) true
#endif

// A launch covers nl links x npl nodes each (node index within the launch
// n = l npl + jn); a single link is nl = 1.
template <typename T> struct KCParams {
    const cx<T>* src;
    long long src_stride;   // elements between consecutive nodes of a link's source (0: shared source)
    long long src_lstride;  // elements between links' sources
    cx<T>* dst;
    long long dst_stride;
    long long dst_lstride;
    const cx<T>* src0;      // if non-null: the source of node jn == 0 of link l is src0 + l src0_lstride
    long long src0_lstride;
    long long N;
    int logN;
    int N1, logN1;
    long long ncols;        // nl * npl * N1 columns in this launch
    int npl;                // nodes per link in this launch
    const NodeC* nodes;     // MPA: constants of link l, node jn at nodes[loff[l] + jn]
    const int* loff;
    NodeC flow;             // SS: constants of the linear step
    unsigned int* err;      // error word of the staged column pass (null: kc_kernel only)
    long long spin_limit;   // polls of each bounded wait of the staged column pass
    // staged column pass only: sources other than src0 (tiled_in) / the
    // destination (tiled_out) hold node spectra in the tile layout (column
    // block b = k1 / G of a node as G x N2 contiguous elements, element
    // (k2, k1 mod G) at b G N2 + k2 G + k1 mod G) instead of natural order
    int tiled_in, tiled_out;
    DbgRange dbg;  // checked range of the debug build
};

template <typename T> struct KRParams {
    cx<T>* data;  // nrows contiguous rows of length N1
    long long nrows;
    long long N;
    int logN;
    int N2;
    T inv_n;  // 1/N
    T rot;    // SS: int sigma over the step
    cx<T>* keep;  // KR_MPA_KEEP: receives A(t), rows laid out as data
    unsigned int* err;       // error word of the staged row pass (null: kr_kernel only)
    long long spin_limit;    // polls of each bounded wait of the staged row pass
    DbgRange dbg;            // checked range of the debug build
};

// Column pass geometry for column length L: G columns per tile, NT threads.
// F: the tiles of field_tiles().
template <typename T, int L, int F = 0> struct KCGeom {
    typedef Tiling<T, F ? F + 2 : 0> P;
    static constexpr bool EX = F > 0 && sizeof(T) == 4;  // FP32 single fields: Tw's EX tables
    static constexpr int G = (P::TE / L) > P::CMIN ? (P::TE / L) : P::CMIN;
    static constexpr int TE = G * L;
    static constexpr int NT = TE / P::E;
    static constexpr int OSH = 5;  // outer-factor two-level split of n2
    static constexpr int OLO = L < 32 ? L : 32;
    static constexpr int OHI = L > 32 ? L / 32 : 1;
    static constexpr size_t smem_elems = (size_t)TE + (TE >> P::PSH) + 1 + Tw<T, L, EX>::N +
                                         (size_t)G * (OLO + OHI);
    static constexpr size_t smem_bytes = smem_elems * sizeof(cx<T>);
};

template <typename T, int L, int F = 0> struct KRGeom {
    typedef Tiling<T, F ? F + 2 : 1> P;
    static constexpr bool EX = F > 0 && sizeof(T) == 4;
    static constexpr int G = (P::TE / L) > 1 ? (P::TE / L) : 1;
    static constexpr int TE = G * L;
    static constexpr int NT = TE / P::E;
    static constexpr int OSH = 7;  // outer-factor split of k1
    static constexpr int OLO = L < 128 ? L : 128;
    static constexpr int OHI = L > 128 ? L / 128 : 1;
    static constexpr size_t smem_elems = (size_t)TE + (TE >> P::PSH) + 1 + Tw<T, L, EX>::N +
                                         (size_t)G * (OLO + OHI);
    static constexpr size_t smem_bytes = smem_elems * sizeof(cx<T>);
};

// 2^-n
template <typename T> __device__ __forceinline__ T pow2_neg(int n) {
    if constexpr (sizeof(T) == 4) return __int_as_float((127 - n) << 23);
    else return __longlong_as_double((long long)(1023 - n) << 52);
}

__device__ __forceinline__ long long signed_k(long long k, long long N) { return k < (N >> 1) ? k : k - N; }

// Global load of data another CTA of the same (persistent) kernel may have
// written: CG = true reads through L2 only (L1 is not coherent within a
// kernel); separate launches use ordinary loads.
template <bool CG, class V> __device__ __forceinline__ V ldx(const V* p) {
    if constexpr (CG) return __ldcg(p);
    else return *p;
}

// Kahan-compensated s += v (c carries the lost low-order part).
template <typename T> __device__ __forceinline__ void kahan_add(T& s, T& c, T v) {
    const T y = v - c;
    const T t = s + y;
    c = (t - s) - y;
    s = t;
}

// L2 prefetch distance of the FP32 column and row passes, in tiles: each CTA
// asks L2 for the tile that the CTA this many launches later will load (0:
// off).  One wave (2 CTAs x 152 SMs) ahead speeds the row pass up by 9 %
// (its tiles are contiguous); the column pass's strided 64-byte rows are
// slower with it.
#ifndef MPA_L2PF_KC
#define MPA_L2PF_KC 0
#endif
// the forward column passes (MPA_POST in the reverse mode's recompute, FWD in
// levels with columns below 2^8) read what the row pass just wrote; one wave
// ahead MPA_POST gains 3.7 % (3815 -> 3957 GB/s at 2^20, 2^12 x 2^8) while the
// inverse pass loses 6.6 % with it.  FWD prefetches only where the node spectra
// exceed L2 (129 MB): two intervals of 143 nodes at 2^17 x 2^7 columns 1075 ->
// 1018 us, of 801 nodes at 2^15 858 -> 820, but 505 -> 512 at 2^16 x 143 (75 MB)
#ifndef MPA_L2PF_KC_POST
#define MPA_L2PF_KC_POST 304
#endif
#ifndef MPA_L2PF_KR
#define MPA_L2PF_KR 304
#endif

__device__ __forceinline__ void prefetch_l2(const void* p, unsigned bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

#ifndef MPA_KC_MINB
#define MPA_KC_MINB 2
#endif
#ifndef MPA_KR_MINB
#define MPA_KR_MINB 2
#endif
template <typename T, int L, int MODE, int F = 0>
__global__ void __launch_bounds__(KCGeom<T, L, F>::NT, KCGeom<T, L, F>::NT <= 256 ? MPA_KC_MINB : 1)
    kc_kernel(const KCParams<T> p) {
    typedef cx<T> C;
    typedef KCGeom<T, L, F> Gm;
    typedef typename Gm::P P;
    constexpr int G = Gm::G, TE = Gm::TE, NT = Gm::NT;
    constexpr bool FWD = (MODE == KC_MPA_POST || MODE == KC_SS_STEP || MODE == KC_FWD || MODE == KC_FWDF || MODE == KC_FWD_T);
    constexpr bool INV = (MODE == KC_MPA_PRE || MODE == KC_SS_STEP || MODE == KC_INV || MODE == KC_INV_T);
    constexpr bool ROWS = (MODE == KC_FWD_T || MODE == KC_INV_T);  // columns are the source's rows
    constexpr bool FAC = (INV || MODE == KC_FWDF) && !ROWS;        // outer factor at the store
    // forward: small radix first, so it ends with an RMAX pass that meets the
    // inverse's first RMAX pass in registers (split-step column pass)
    typedef Xform<T, L, G, NT, P::RMAX, +1, LAYOUT_COL, P::PSH, true, 0, false, Gm::EX> XF;
    typedef Xform<T, L, G, NT, P::RMAX, -1, LAYOUT_COL, P::PSH, false, 0, false, Gm::EX> XI;
    static_assert(!(FWD && INV) || XF::RL == XI::R0, "forward/inverse junction radix");
    typedef typename std::conditional<FWD, XF, XI>::type XA;  // first transform
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* s = reinterpret_cast<C*>(smem_raw);
    C* thi = s + TE + (TE >> P::PSH) + 1;
    C* tlo = thi + TwDims<L>::NHI;
    C* olo = thi + Tw<T, L, Gm::EX>::N;  // [OLO][G]
    C* ohi = olo + G * Gm::OLO;     // [OHI][G]
    const int tid = threadIdx.x;
    const long long col0 = (long long)blockIdx.x * G;
    const int N1m = p.N1 - 1;
    constexpr bool FAST = sizeof(T) == 4;  // FP32: finite-difference phases + polynomial exp

    // passes that a scan follows let it start only at their end (pdl_go)
    constexpr bool EARLY = F > 0 || MODE == KC_MPA_PRE || MODE == KC_INV;
    if constexpr (EARLY) pdl_go();
    tw_init<T, L, Gm::EX>(thi, tlo, tid, NT);
    if constexpr (FAC) {
        // W_N^{-n2 k1} for the tile's columns: olo[m][g] = W^{-k1 m}, ohi[h][g] = W^{-k1 32 h} (FWDF: +)
        for (int i = tid; i < G * (Gm::OLO + Gm::OHI); i += NT) {
            const int g = i % G, m = i / G;
            const long long k1 = MODE == KC_FWDF ? -((col0 + g) & N1m) : (col0 + g) & N1m;
            if (m < Gm::OLO) olo[m * G + g] = expi_ratio<T>(-k1 * m, p.logN);
            else ohi[(m - Gm::OLO) * G + g] = expi_ratio<T>(-k1 * ((long long)(m - Gm::OLO) << Gm::OSH), p.logN);
        }
    }
    __syncthreads();
    pdl_wait();

    // ---- load: element j + r L/R0 of column col0 + g, straight into registers
    C vin[XA::Q0][XA::R0];
#pragma unroll
    for (int q = 0; q < XA::Q0; ++q) {
        int j, g;
        bmap<LAYOUT_COL, L, G, XA::R0>(tid + q * NT, j, g);
        const long long col = col0 + g;
        const bool ok = col < p.ncols;
        const int node = ok ? (int)(col >> p.logN1) : 0;
        const int l = node / p.npl, jn = node - l * p.npl;
        const long long c = col & N1m;
        const C* src = ROWS                  ? p.src + col * L
                       : (p.src0 && jn == 0) ? p.src0 + l * p.src0_lstride + c
                                             : p.src + l * p.src_lstride + jn * p.src_stride + c;
        const long long rs = ROWS ? 1 : p.N1;  // distance of the column's rows
        NodeC nc{};
        if constexpr (MODE == KC_MPA_PRE) {
            if (MPA_DBG_OK(p.dbg, p.loff + l, sizeof(int)) && MPA_DBG_OK(p.dbg, p.nodes + p.loff[l] + jn, sizeof(NodeC)))
                nc = p.nodes[p.loff[l] + jn];
        }
        unsigned long long th[XA::R0];
        if constexpr (FAST && MODE == KC_MPA_PRE)
            phase_run<XA::R0>(c + (long long)j * p.N1, (long long)p.N1 * (L / XA::R0), nc, th);
        [[maybe_unused]] C odd = mkc(T(0), T(0));
#pragma unroll
        for (int r = 0; r < XA::R0; ++r) {
            const int row = j + r * (L / XA::R0);
            C v = ok && MPA_DBG_OK(p.dbg, src + row * rs, sizeof(C)) ? src[row * rs] : mkc(T(0), T(0));
            if constexpr (MODE == KC_MPA_PRE) {
                // MPA step 2: A_hat_j = psi_j exp(i beta(w, z_j) + int G)
                C ph;
                if constexpr (FAST) ph = expi_pair(th, r, odd);
                else ph = expi_at<T, L>(phase_q64(signed_k(c + (long long)row * p.N1, p.N), nc), thi);
                v = cscale(cmul(v, ph), (T)nc.pre);
            }
            vin[q][r] = v;
        }
    }

    constexpr bool LEVEL_FWD = F == 0 && MODE == KC_FWD;  // (or a single field beyond 2^22: no error word)
    constexpr int L2PF = MODE == KC_MPA_POST || LEVEL_FWD ? MPA_L2PF_KC_POST : MPA_L2PF_KC;
    if constexpr (FAST && L2PF > 0) {
        const long long tb = (long long)blockIdx.x + L2PF;
        if (tb < (long long)gridDim.x && (!LEVEL_FWD || (p.err && p.ncols * L > (1ll << 24)))) {
            // the first node's columns of that tile (all of it when G <= N1)
            const long long col = tb * G;
            const int node = (int)(col >> p.logN1);
            const int l = node / p.npl, jn = node - l * p.npl;
            const long long c = col & N1m;
            const C* src = (p.src0 && jn == 0) ? p.src0 + l * p.src0_lstride + c
                                               : p.src + l * p.src_lstride + jn * p.src_stride + c;
            long long w = p.ncols - col < G ? p.ncols - col : G;
            if (w > p.N1 - c) w = p.N1 - c;
            // whole 128-byte L2 lines: a tile narrower than a line prefetches
            // the line once (the tile at its start), the others skip
            constexpr long long LINE = 128 / (long long)sizeof(C);
            bool go = true;
            if (w < LINE) {
                go = (c % LINE) == 0 && c + LINE <= p.N1;
                w = LINE;
            }
            if (go)
                for (int r = tid; r < L; r += NT) prefetch_l2(src + (long long)r * p.N1, (unsigned)(w * sizeof(C)));
        }
    }

    // ---- transforms
    constexpr int QO = INV ? XI::QL : XF::QL, RO = INV ? XI::RL : XF::RL;
    C vout[QO][RO];
    if constexpr (FWD && INV) {
        C vm[XF::QL][XF::RL];
        XF::run(vin, vm, s, thi, tlo);
        // exact linear step exp(i beta(w; za, zb) + int G) between the kicks of Eq. (4)
#pragma unroll
        for (int q = 0; q < XF::QL; ++q) {
            int j, g;
            bmap<LAYOUT_COL, L, G, XF::RL>(tid + q * NT, j, g);
            const long long c = (col0 + g) & N1m;
            unsigned long long th[XF::RL];
            if constexpr (FAST) phase_run<XF::RL>(c + (long long)j * p.N1, (long long)p.N1 * (L / XF::RL), p.flow, th);
            [[maybe_unused]] C odd = mkc(T(0), T(0));
#pragma unroll
            for (int r = 0; r < XF::RL; ++r) {
                const int row = j + r * (L / XF::RL);
                C ph;
                if constexpr (FAST) ph = expi_pair(th, r, odd);
                else ph = expi_at<T, L>(phase_q64(signed_k(c + (long long)row * p.N1, p.N), p.flow), thi);
                vm[q][r] = cscale(cmul(vm[q][r], ph), (T)p.flow.pre);
            }
        }
        XI::run(vm, vout, s, thi, tlo);
    } else if constexpr (FWD) {
        XF::run(vin, vout, s, thi, tlo);
    } else {
        XI::run(vin, vout, s, thi, tlo);
    }

    if constexpr (!EARLY) pdl_go();
    // ---- epilogue and store: element j + r L/RO of column col0 + g
#pragma unroll
    for (int q = 0; q < QO; ++q) {
        int j, g;
        bmap<LAYOUT_COL, L, G, RO>(tid + q * NT, j, g);
        const long long col = col0 + g;
        if (col >= p.ncols) continue;
        const int node = (int)(col >> p.logN1);
        const int l = node / p.npl, jn = node - l * p.npl;
        const long long c = col & N1m;
        C* dst = p.dst + l * p.dst_lstride + jn * p.dst_stride + c;
        NodeC nc{};
        if constexpr (MODE == KC_MPA_POST) {
            if (MPA_DBG_OK(p.dbg, p.loff + l, sizeof(int)) && MPA_DBG_OK(p.dbg, p.nodes + p.loff[l] + jn, sizeof(NodeC)))
                nc = p.nodes[p.loff[l] + jn];
        }
        unsigned long long th[RO];
        if constexpr (FAST && MODE == KC_MPA_POST)
            phase_run<RO>(c + (long long)j * p.N1, (long long)p.N1 * (L / RO), nc, th);
        // rows j + r L/RO share their low outer-factor index when L/RO is a
        // multiple of the low table's length: one lookup per butterfly
        constexpr bool HOIST = (L / RO) % Gm::OLO == 0;
        C wlo = mkc(T(1), T(0));
        if constexpr (FAC && HOIST) wlo = olo[(j & (Gm::OLO - 1)) * G + g];
        [[maybe_unused]] C odd = mkc(T(0), T(0));
#pragma unroll
        for (int r = 0; r < RO; ++r) {
            const int row = j + r * (L / RO);
            C v = vout[q][r];
            if constexpr (FAC) {
                // four-step factor W_N^{-n2 k1}, n2 = row
                C w = HOIST ? wlo : olo[(row & (Gm::OLO - 1)) * G + g];
                if constexpr (Gm::OHI > 1) w = cmul(ohi[(row >> Gm::OSH) * G + g], w);
                v = cmul(v, w);
            }
            if constexpr (MODE == KC_INV_T) v = cscale(v, pow2_neg<T>(p.logN));
            if constexpr (MODE == KC_MPA_POST) {
                // V_j = sigma(z_j) dz F[|A_j|^2 A_j] exp(-i beta(w, z_j) - int G)   (Eq. (6))
                C ph;
                if constexpr (FAST) ph = expi_pair(th, r, odd);
                else ph = expi_at<T, L>(phase_q64(signed_k(c + (long long)row * p.N1, p.N), nc), thi);
                v = cscale(cmul(v, cconj(ph)), (T)nc.post);
            }
            if (MPA_DBG_OK(p.dbg, dst + (long long)row * p.N1, sizeof(C))) dst[(long long)row * p.N1] = v;
        }
    }
}

template <typename T, int L, int MODE, int F = 0>
__global__ void __launch_bounds__(KRGeom<T, L, F>::NT, KRGeom<T, L, F>::NT <= 256 ? MPA_KR_MINB : 1)
    kr_kernel(const KRParams<T> p) {
    typedef cx<T> C;
    typedef KRGeom<T, L, F> Gm;
    typedef typename Gm::P P;
    constexpr int G = Gm::G, TE = Gm::TE, NT = Gm::NT;
    constexpr bool INV = (MODE != KR_FWD);
    constexpr bool FWD = (MODE != KR_INV);
    // inverse: small radix last, forward: small radix first, so the two meet
    // in registers around the pointwise step
    typedef Xform<T, L, G, NT, P::RMAX, -1, LAYOUT_ROW, P::PSH, false, 0, false, Gm::EX> XI;
    typedef Xform<T, L, G, NT, P::RMAX, +1, LAYOUT_ROW, P::PSH, true, 0, false, Gm::EX> XF;
    static_assert(!(FWD && INV) || XI::RL == XF::R0, "inverse/forward junction radix");
    typedef typename std::conditional<INV, XI, XF>::type XA;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* s = reinterpret_cast<C*>(smem_raw);
    C* thi = s + TE + (TE >> P::PSH) + 1;
    C* tlo = thi + TwDims<L>::NHI;
    C* olo = thi + Tw<T, L, Gm::EX>::N;  // [G][OLO]
    C* ohi = olo + G * Gm::OLO;     // [G][OHI]
    const int tid = threadIdx.x;
    const long long row0 = (long long)blockIdx.x * G;

    pdl_go();
    tw_init<T, L, Gm::EX>(thi, tlo, tid, NT);
    if constexpr (FWD) {
        // W_N^{+n2 k1} for the tile's rows: olo[g][m] = W^{n2 m}, ohi[g][h] = W^{n2 128 h}
        for (int i = tid; i < G * (Gm::OLO + Gm::OHI); i += NT) {
            const int g = i / (Gm::OLO + Gm::OHI), m = i % (Gm::OLO + Gm::OHI);
            const long long n2 = (row0 + g) & (p.N2 - 1);
            if (m < Gm::OLO) olo[g * Gm::OLO + m] = expi_ratio<T>(n2 * m, p.logN);
            else ohi[g * Gm::OHI + (m - Gm::OLO)] = expi_ratio<T>(n2 * ((long long)(m - Gm::OLO) << Gm::OSH), p.logN);
        }
    }
    __syncthreads();
    pdl_wait();

    C vin[XA::Q0][XA::R0];
#pragma unroll
    for (int q = 0; q < XA::Q0; ++q) {
        int j, g;
        bmap<LAYOUT_ROW, L, G, XA::R0>(tid + q * NT, j, g);
        const bool ok = row0 + g < p.nrows;
        const C* src = p.data + (row0 + g) * L;
#pragma unroll
        for (int r = 0; r < XA::R0; ++r)
            vin[q][r] = ok && MPA_DBG_OK(p.dbg, src + j + r * (L / XA::R0), sizeof(C)) ? src[j + r * (L / XA::R0)]
                                                                                     : mkc(T(0), T(0));
    }

    if constexpr (F == 0 && sizeof(T) == 4 && MPA_L2PF_KR > 0) {
        const long long tb = (long long)blockIdx.x + MPA_L2PF_KR;
        const long long r0 = tb * G;
        if (tb < (long long)gridDim.x && r0 < p.nrows) {
            const long long nr = p.nrows - r0 < G ? p.nrows - r0 : G;
            const long long bytes = nr * L * (long long)sizeof(C);  // contiguous rows
            const C* base = p.data + r0 * L;
            for (long long o = (long long)tid * 256; o < bytes; o += (long long)NT * 256)
                prefetch_l2(reinterpret_cast<const char*>(base) + o, (unsigned)(bytes - o < 256 ? bytes - o : 256));
        }
    }

    constexpr int QO = FWD ? XF::QL : XI::QL, RO = FWD ? XF::RL : XI::RL;
    C vout[QO][RO];
    if constexpr (INV && FWD) {
        C vm[XI::QL][XI::RL];
        XI::run(vin, vm, s, thi, tlo);
#pragma unroll
        for (int q = 0; q < XI::QL; ++q) {
            C* kp = nullptr;
            int jk = 0;
            if constexpr (MODE == KR_MPA_KEEP) {
                int g;
                bmap<LAYOUT_ROW, L, G, XI::RL>(tid + q * NT, jk, g);
                if (row0 + g < p.nrows) kp = p.keep + (row0 + g) * L;
            }
#pragma unroll
            for (int r = 0; r < XI::RL; ++r) {
                C a = cscale(vm[q][r], p.inv_n);  // A(t) (MPA step 3 / SS inverse)
                if constexpr (MODE == KR_MPA_KEEP) {
                    if (kp && MPA_DBG_OK(p.dbg, kp + jk + r * (L / XI::RL), sizeof(C))) kp[jk + r * (L / XI::RL)] = a;
                }
                const T pw = a.x * a.x + a.y * a.y;
                if constexpr (MODE == KR_MPA || MODE == KR_MPA_KEEP) {
                    a = cscale(a, pw);  // |A|^2 A (MPA step 4)
                } else {
                    T sn, cs;  // A exp(i s |A|^2), the nonlinear step of Eq. (4)
                    sincos_kerr(p.rot * pw, &sn, &cs);
                    a = cmul(a, mkc(cs, sn));
                }
                vm[q][r] = a;
            }
        }
        XF::run(vm, vout, s, thi, tlo);
    } else if constexpr (INV) {
        XI::run(vin, vout, s, thi, tlo);
    } else {
        XF::run(vin, vout, s, thi, tlo);
    }

#pragma unroll
    for (int q = 0; q < QO; ++q) {
        int j, g;
        bmap<LAYOUT_ROW, L, G, RO>(tid + q * NT, j, g);
        if (row0 + g >= p.nrows) continue;
        C* dst = p.data + (row0 + g) * L;
        constexpr bool HOIST = (L / RO) % Gm::OLO == 0;  // one low-table lookup per butterfly
        C wlo = mkc(T(1), T(0));
        if constexpr (FWD && HOIST) wlo = olo[g * Gm::OLO + (j & (Gm::OLO - 1))];
#pragma unroll
        for (int r = 0; r < RO; ++r) {
            const int l = j + r * (L / RO);  // k1
            C v = vout[q][r];
            if constexpr (FWD) {
                C w = HOIST ? wlo : olo[g * Gm::OLO + (l & (Gm::OLO - 1))];
                if constexpr (Gm::OHI > 1) w = cmul(ohi[g * Gm::OHI + (l >> Gm::OSH)], w);
                v = cmul(v, w);
            } else {
                v = cscale(v, p.inv_n);
            }
            if (MPA_DBG_OK(p.dbg, dst + l, sizeof(C))) dst[l] = v;
        }
    }
}

// ------------------------------------------------------------------
// Whole node transform on chip (MPA steps 2-4 and the weight of Eq. (6)) for
// N small enough that one spectrum fits in a CTA's shared memory (N <= 2^14
// FP32, 2^13 FP64): G = TE/N nodes per CTA, each a row of the row-pass tile
// layout holding its spectrum in natural order:
//   A_hat = psi_j exp(i beta_j + int G)        (phase at the load, step 2; PIN)
//   A = F^-1[A_hat]; U = |A|^2 A; F[U]          (steps 3-4, in shared memory)
//   V_j = F[U] sigma_j dz exp(-i beta_j - int G)   (at the store, Eq. (6); POUT)
// Without PIN the source holds A_hat_j already, without POUT the destination
// receives F[U] (ScanParams::phases: the scan applies the phases).
// One HBM (or L2) round trip per node instead of the three of the column,
// row and column passes, no four-step outer factors.  Node addressing as in
// KCParams (nl links x npl nodes, psi_0 shared by node 0).
template <typename T> struct KNParams {
    const cx<T>* src;
    long long src_stride, src_lstride;
    const cx<T>* src0;  // if non-null: the source of node jn == 0 of link l is src0 + l src0_lstride
    long long src0_lstride;
    cx<T>* dst;
    long long dst_stride, dst_lstride;
    long long nrows;    // nl * npl nodes in this launch
    int npl;
    const NodeC* nodes;  // link l, node jn at nodes[loff[l] + jn]
    const int* loff;
    T inv_n;
    bool phase_in, phase_out;  // kn_launch: the phases applied at the load and at the store
    DbgRange dbg;  // checked range of the debug build
};

// F = 1 (FP32): one node a CTA (several below 2^10 modes), 16 elements a
// thread, for launches whose large tiles would not fill the SMs twice (kn_fine).
template <typename T, int L, int F = 0> struct KNGeom {
    typedef KRGeom<T, L> R;
    typedef Tiling<T, F ? 5 : 1> P;
    static constexpr bool EX = F > 0 && sizeof(T) == 4 && L <= 2048;
    static constexpr int G = F ? (L >= 1024 ? 1 : 1024 / L) : R::G, TE = G * L, NT = TE / P::E;
    static constexpr size_t smem_bytes = ((size_t)TE + (TE >> P::PSH) + 1 + Tw<T, L, EX>::N) * sizeof(cx<T>);
};

// The node rows row0 .. row0 + G - 1 of a launch (one tile) through steps
// 2-4 and the weight of Eq. (6); the block's threads and shared memory.
template <typename T, int L, bool CG, bool PIN, bool POUT, int F = 0>
__device__ __forceinline__ void kn_tile(const KNParams<T>& p, long long row0, unsigned char* smem_raw) {
    typedef cx<T> C;
    typedef KNGeom<T, L, F> Gm;
    typedef typename Gm::P P;
    constexpr int G = Gm::G, NT = Gm::NT, TE = Gm::TE;
    typedef Xform<T, L, G, NT, P::RMAX, -1, LAYOUT_ROW, P::PSH, false, 0, false, Gm::EX> XI;
    typedef Xform<T, L, G, NT, P::RMAX, +1, LAYOUT_ROW, P::PSH, true, 0, false, Gm::EX> XF;
    static_assert(XI::RL == XF::R0, "inverse/forward junction radix");
    constexpr bool FAST = sizeof(T) == 4;  // FP32: finite-difference phases + polynomial exp
    C* s = reinterpret_cast<C*>(smem_raw);
    C* thi = s + TE + (TE >> P::PSH) + 1;
    C* tlo = thi + TwDims<L>::NHI;
    const int tid = threadIdx.x;

    tw_init<T, L, Gm::EX>(thi, tlo, tid, NT);
    __syncthreads();
    if constexpr (!CG) pdl_wait();  // CG: called inside the persistent kernel

    // ---- load node spectra (natural order, k = element index) and step 2
    C vin[XI::Q0][XI::R0];
#pragma unroll
    for (int q = 0; q < XI::Q0; ++q) {
        int j, g;
        bmap<LAYOUT_ROW, L, G, XI::R0>(tid + q * NT, j, g);
        const long long row = row0 + g;
        const bool ok = row < p.nrows;
        const int node = ok ? (int)row : 0;
        const int l = node / p.npl, jn = node - l * p.npl;
        const C* src = (p.src0 && jn == 0) ? p.src0 + l * p.src0_lstride : p.src + l * p.src_lstride + jn * p.src_stride;
        if constexpr (!PIN) {
#pragma unroll
            for (int r = 0; r < XI::R0; ++r) {
                const int k = j + r * (L / XI::R0);
                vin[q][r] = ok && MPA_DBG_OK(p.dbg, src + k, sizeof(C)) ? ldx<CG>(src + k) : mkc(T(0), T(0));
            }
            continue;
        }
        NodeC nc{};
        if (MPA_DBG_OK(p.dbg, p.loff + l, sizeof(int)) && MPA_DBG_OK(p.dbg, p.nodes + p.loff[l] + jn, sizeof(NodeC)))
            nc = p.nodes[p.loff[l] + jn];
        unsigned long long th[XI::R0];
        if constexpr (FAST) phase_run<XI::R0>(j, L / XI::R0, nc, th);
        C odd = mkc(T(0), T(0));
#pragma unroll
        for (int r = 0; r < XI::R0; ++r) {
            const int k = j + r * (L / XI::R0);
            C v = ok && MPA_DBG_OK(p.dbg, src + k, sizeof(C)) ? ldx<CG>(src + k) : mkc(T(0), T(0));
            C ph;
            if constexpr (FAST) ph = expi_pair(th, r, odd);
            else ph = expi_at<T, L>(phase_q64(signed_k(k, L), nc), thi);
            vin[q][r] = cscale(cmul(v, ph), (T)nc.pre);
        }
    }

    // ---- steps 3-4: inverse transform, 1/N, |A|^2 A, forward transform
    C vm[XI::QL][XI::RL];
    XI::run(vin, vm, s, thi, tlo);
#pragma unroll
    for (int q = 0; q < XI::QL; ++q) {
#pragma unroll
        for (int r = 0; r < XI::RL; ++r) {
            const C a = cscale(vm[q][r], p.inv_n);
            vm[q][r] = cscale(a, a.x * a.x + a.y * a.y);
        }
    }
    C vout[XF::QL][XF::RL];
    XF::run(vm, vout, s, thi, tlo);

    if constexpr (!CG) pdl_go();
    // ---- V_j (Eq. (6)) and the store, natural order
#pragma unroll
    for (int q = 0; q < XF::QL; ++q) {
        int j, g;
        bmap<LAYOUT_ROW, L, G, XF::RL>(tid + q * NT, j, g);
        const long long row = row0 + g;
        if (row >= p.nrows) continue;
        const int node = (int)row;
        const int l = node / p.npl, jn = node - l * p.npl;
        C* dst = p.dst + l * p.dst_lstride + jn * p.dst_stride;
        if constexpr (!POUT) {
#pragma unroll
            for (int r = 0; r < XF::RL; ++r) {
                const int k = j + r * (L / XF::RL);
                if (MPA_DBG_OK(p.dbg, dst + k, sizeof(C))) dst[k] = vout[q][r];
            }
            continue;
        }
        NodeC nc{};
        if (MPA_DBG_OK(p.dbg, p.loff + l, sizeof(int)) && MPA_DBG_OK(p.dbg, p.nodes + p.loff[l] + jn, sizeof(NodeC)))
            nc = p.nodes[p.loff[l] + jn];
        unsigned long long th[XF::RL];
        if constexpr (FAST) phase_run<XF::RL>(j, L / XF::RL, nc, th);
        C odd = mkc(T(0), T(0));
#pragma unroll
        for (int r = 0; r < XF::RL; ++r) {
            const int k = j + r * (L / XF::RL);
            C ph;
            if constexpr (FAST) ph = expi_pair(th, r, odd);
            else ph = expi_at<T, L>(phase_q64(signed_k(k, L), nc), thi);
            if (MPA_DBG_OK(p.dbg, dst + k, sizeof(C))) dst[k] = cscale(cmul(vout[q][r], cconj(ph)), (T)nc.post);
        }
    }
}

template <typename T, int L, bool PIN, bool POUT, int F = 0>
__global__ void __launch_bounds__(KNGeom<T, L, F>::NT, KNGeom<T, L, F>::NT <= 256 ? MPA_KR_MINB : 1)
    kn_kernel(const KNParams<T> p) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    kn_tile<T, L, false, PIN, POUT, F>(p, (long long)blockIdx.x * KNGeom<T, L, F>::G, smem_raw);
}

// ------------------------------------------------------------------
// Wavefront column pass (FP32): one CTA owns one column tile of one block
// of B consecutive nodes at one Picard level and walks the nodes in order:
//   forward column DFTs (finishing F[|A_j|^2 A_j])
//   V_j = F[...] exp(-i beta_j) sigma_j dz / exp(int G)          (Eq. (6))
//   psi^{(n+1)}_j = psi_0 + i (R + V_j/2),  R += V_j              (step 5)
//   A_hat = psi^{(n+1)}_j exp(i beta_j + int G) and the inverse column DFTs
//   of level n+1 (steps 2-3), written back over the node's buffer.
// R (the trapezoid running sum of this level, Kahan-compensated, the
// compensation kept in shared memory) persists across the block in
// registers and across blocks in global memory.  The phase of node j is
// evaluated once for both directions.  On the last level the inverse
// transform is instead that of the next block's first iteration for the
// node S B further on (psi_0 exp(i beta + int G)), and the node-M value
// psi_0 + i (R + V_M/2) is emitted in FP64 for step 7.
struct KCWJob {
    int level, slot, node_first, n_nodes, head_first, n_head, last;
};

struct KCWParams {
    float2* work;           // slots of B node buffers
    long long slot_stride;  // elements between slots
    long long N;
    int logN, N1, logN1, M;
    const NodeC* nodes;     // this interval's constants, node j at nodes[j]
    const float2* psi0;     // psi_0 (complex64, natural order)
    const float2* v0;       // V_0 (complex64) for blocks that start at node 1
    float2* Rg;             // [levels][N] running sums
    float2* Cg;             // [levels][N] Kahan compensations
    double2* D;             // R + V_M/2 at node M (so psi_M = psi_0 + i D), FP64
    int n_jobs;
    KCWJob job[8];  // one per Picard level (n_iter <= 8)
};

// Tile of the wavefront column pass: MPA_KCW_TE elements (at least 4
// columns); the running sums and compensations take 16 bytes per element of
// shared memory, so 4096-element tiles (about 102 KB with the transform
// tile) let two CTAs share an SM and 8192-element ones (about 200 KB) one.
#ifndef MPA_KCW_TE
#define MPA_KCW_TE 4096
#endif
#ifndef MPA_KCW_MINB
#define MPA_KCW_MINB 2
#endif
template <int L> struct KCWGeom {
    typedef Tiling<float, 2> P;
    static constexpr int G = (MPA_KCW_TE / L) > 4 ? (MPA_KCW_TE / L) : 4, TE = G * L, NT = TE / P::E;
    static constexpr int OSH = 5, OLO = L < 32 ? L : 32, OHI = L > 32 ? L / 32 : 1;
    // float2 offset of the running sums (float4 per element): rounded up to
    // an even count so the array starts on a 16-byte boundary
    static constexpr size_t RC_OFF =
        (((size_t)TE + (TE >> P::PSH) + 1 + TwDims<L>::NLO + TwDims<L>::NHI + (size_t)G * (OLO + OHI)) + 1) & ~(size_t)1;
    static constexpr size_t smem_bytes = RC_OFF * sizeof(float2) + (size_t)TE * sizeof(float4);
};

// The node loop of one job; LAST selects the last Picard level (heads of
// the next blocks instead of the next level, and the node-M output).
template <int L, bool LAST>
__device__ __forceinline__ void kcw_job(const KCWParams& p, const KCWJob& job, float2* s, const float2* thi,
                                        const float2* tlo, const float2* olo, const float2* ohi, float4* rc,
                                        int col0) {
    typedef float2 C;
    typedef KCWGeom<L> Gm;
    typedef Tiling<float, 2> P;
    constexpr int G = Gm::G, NT = Gm::NT;
    typedef Xform<float, L, G, NT, P::RMAX, +1, LAYOUT_COL, P::PSH, true> XF;
    typedef Xform<float, L, G, NT, P::RMAX, -1, LAYOUT_COL, P::PSH, false> XI;
    constexpr int QJ = XF::QL, RJ = XF::RL;
    const int tid = threadIdx.x;
    const long long N = p.N;
    const long long D = (long long)p.N1 * (L / RJ);

    // running sums of this level (and Kahan compensations) for the thread's
    // junction elements, kept in shared memory across the node loop
#pragma unroll
    for (int q = 0; q < QJ; ++q) {
        int j, g;
        bmap<LAYOUT_COL, L, G, RJ>(tid + q * NT, j, g);
#pragma unroll
        for (int r = 0; r < RJ; ++r) {
            const long long k = (col0 + g) + (long long)(j + r * (L / RJ)) * p.N1;
            float4 e;
            if (job.node_first == 1) {
                const float2 v = p.v0[k];
                e = make_float4(0.5f * v.x, 0.5f * v.y, 0.f, 0.f);  // V_0 / 2
            } else {
                const float2 rv = p.Rg[(long long)job.level * N + k], cv = p.Cg[(long long)job.level * N + k];
                e = make_float4(rv.x, rv.y, cv.x, cv.y);
            }
            rc[(q * RJ + r) * NT + tid] = e;
        }
    }

    float2* slot = p.work + (long long)job.slot * p.slot_stride;
    for (int i = 0; i < job.n_nodes; ++i) {
        const int jn = job.node_first + i;
        float2* buf = slot + (long long)i * N;
        // ---- forward column DFTs of node jn (first pass straight from global)
        C vin[XF::Q0][XF::R0];
#pragma unroll
        for (int q = 0; q < XF::Q0; ++q) {
            int j, g;
            bmap<LAYOUT_COL, L, G, XF::R0>(tid + q * NT, j, g);
            const C* src = buf + col0 + g;
#pragma unroll
            for (int r = 0; r < XF::R0; ++r) vin[q][r] = src[(long long)(j + r * (L / XF::R0)) * p.N1];
        }
        C v[QJ][RJ];
        XF::run(vin, v, s, thi, tlo);
        const bool head = LAST && i < job.n_head;
        const NodeC nc = p.nodes[jn];
        const float post = (float)nc.post;
#pragma unroll
        for (int q = 0; q < QJ; ++q) {
            int j, g;
            bmap<LAYOUT_COL, L, G, RJ>(tid + q * NT, j, g);
            const long long c = col0 + g;
            // elements in s order: s = -RJ/2 .. RJ/2-1, r = (s + RJ) mod RJ, k' = c + N1 (j + s L/RJ)
            const long long kf = c + (long long)p.N1 * j - (long long)(RJ / 2) * D;
            PhaseRun pr(kf, D, nc);
            if constexpr (!LAST) {
                const float pre = (float)nc.pre;
#pragma unroll
                for (int t = 0; t < RJ; ++t) {
                    const int r = (t + RJ / 2) % RJ;
                    const long long k = c + (long long)(j + r * (L / RJ)) * p.N1;
                    const C ph = expi_turns_poly(pr.next());
                    // V_j (Eq. (6)) and psi^{(n+1)}_j = psi_0 + i (R + V_j/2) (step 5)
                    const C V = cscale(cmul(v[q][r], cconj(ph)), post);
                    float4 e = rc[(q * RJ + r) * NT + tid];  // (R, compensation)
                    const float2 p0 = p.psi0[k];
                    const float sx = (e.x - e.z) + 0.5f * V.x, sy = (e.y - e.w) + 0.5f * V.y;
                    kahan_add(e.x, e.z, V.x);
                    kahan_add(e.y, e.w, V.y);
                    rc[(q * RJ + r) * NT + tid] = e;
                    // step 2 of the next iteration at the same node
                    v[q][r] = cscale(cmul(make_float2(p0.x - sy, p0.y + sx), ph), pre);
                }
            } else {
#pragma unroll
                for (int t = 0; t < RJ; ++t) {
                    const int r = (t + RJ / 2) % RJ;
                    const C ph = expi_turns_poly(pr.next());
                    const C V = cscale(cmul(v[q][r], cconj(ph)), post);
                    float4 e = rc[(q * RJ + r) * NT + tid];  // (R, compensation)
                    if (jn == p.M) {
                        // R + V_M/2 before adding V_M: psi_M = psi_0 + i D (FP64)
                        const long long k = c + (long long)(j + r * (L / RJ)) * p.N1;
                        p.D[k] = make_double2(((double)e.x - (double)e.z) + 0.5 * (double)V.x,
                                              ((double)e.y - (double)e.w) + 0.5 * (double)V.y);
                    }
                    kahan_add(e.x, e.z, V.x);
                    kahan_add(e.y, e.w, V.y);
                    rc[(q * RJ + r) * NT + tid] = e;
                }
                if (head) {
                    // first iteration of the node S B further on: psi_0 exp(i beta + int G)
                    const NodeC nh = p.nodes[job.head_first + i];
                    const float preh = (float)nh.pre;
                    PhaseRun ph2(kf, D, nh);
#pragma unroll
                    for (int t = 0; t < RJ; ++t) {
                        const int r = (t + RJ / 2) % RJ;
                        const long long k = c + (long long)(j + r * (L / RJ)) * p.N1;
                        v[q][r] = cscale(cmul(p.psi0[k], expi_turns_poly(ph2.next())), preh);
                    }
                }
            }
        }
        if (!LAST || head) {
            // ---- inverse column DFTs, four-step factor, store over the node buffer
            C vo[XI::QL][XI::RL];
            XI::run(v, vo, s, thi, tlo);
#pragma unroll
            for (int q = 0; q < XI::QL; ++q) {
                int j, g;
                bmap<LAYOUT_COL, L, G, XI::RL>(tid + q * NT, j, g);
                C* dst = buf + col0 + g;
#pragma unroll
                for (int r = 0; r < XI::RL; ++r) {
                    const int row = j + r * (L / XI::RL);
                    C w = olo[(row & (Gm::OLO - 1)) * G + g];
                    if constexpr (Gm::OHI > 1) w = cmul(ohi[(row >> Gm::OSH) * G + g], w);
                    dst[(long long)row * p.N1] = cmul(vo[q][r], w);
                }
            }
        }
    }

    // ---- running sums back to global memory for the next block
#pragma unroll
    for (int q = 0; q < QJ; ++q) {
        int j, g;
        bmap<LAYOUT_COL, L, G, RJ>(tid + q * NT, j, g);
#pragma unroll
        for (int r = 0; r < RJ; ++r) {
            const long long k = (col0 + g) + (long long)(j + r * (L / RJ)) * p.N1;
            const float4 e = rc[(q * RJ + r) * NT + tid];
            p.Rg[(long long)job.level * N + k] = make_float2(e.x, e.y);
            p.Cg[(long long)job.level * N + k] = make_float2(e.z, e.w);
        }
    }
}

template <int L>
__global__ void __launch_bounds__(KCWGeom<L>::NT, KCWGeom<L>::NT <= 256 ? MPA_KCW_MINB : 1)
    kcw_kernel(const KCWParams p) {
    typedef float2 C;
    typedef KCWGeom<L> Gm;
    typedef Tiling<float, 2> P;
    constexpr int G = Gm::G, TE = Gm::TE, NT = Gm::NT;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* s = reinterpret_cast<C*>(smem_raw);
    C* thi = s + TE + (TE >> P::PSH) + 1;
    C* tlo = thi + TwDims<L>::NHI;
    C* olo = tlo + TwDims<L>::NLO;  // [OLO][G]
    C* ohi = olo + G * Gm::OLO;     // [OHI][G]
    float4* rc = reinterpret_cast<float4*>(s + Gm::RC_OFF);  // [E][NT] (R, compensation), 16-B aligned
    const int tid = threadIdx.x;
    const KCWJob job = p.job[blockIdx.y];
    const int col0 = blockIdx.x * G;  // column within a node (tiles never straddle nodes)

    tw_init<float, L>(thi, tlo, tid, NT);
    for (int i = tid; i < G * (Gm::OLO + Gm::OHI); i += NT) {
        const int g = i % G, m = i / G;
        const long long k1 = col0 + g;
        if (m < Gm::OLO) olo[m * G + g] = expi_ratio<float>(-k1 * m, p.logN);
        else ohi[(m - Gm::OLO) * G + g] = expi_ratio<float>(-k1 * ((long long)(m - Gm::OLO) << Gm::OSH), p.logN);
    }
    __syncthreads();
    if (job.last) kcw_job<L, true>(p, job, s, thi, tlo, olo, ohi, rc, col0);
    else kcw_job<L, false>(p, job, s, thi, tlo, olo, ohi, rc, col0);
}

// Eq. (6) for every frequency k: running trapezoid sum over nodes j = 1..M
//   psi^{(n+1)}_l = psi_0 + i (V_0/2 + sum_{j=1}^{l-1} V_j + V_l/2),
// with V_j stored in psi[j] (node 0 holds V_0).  FP32 sums are Kahan-
// compensated; the final value at node M is formed in FP64.
//   mode 0: write psi^{(n+1)}_j into psi[j], j >= 1 (next iteration)
// With `phases`, psi[j] holds F_j = F[|A_j|^2 A_j] instead, the scan forms
// V_j = sigma_j dz F_j exp(-i beta_j - int G) itself, and mode 0 writes
// A_hat^{(n+1)}_j = psi^{(n+1)}_j exp(i beta_j + int G).
//   mode 1: step 7: state <- psi_M exp(i beta(w, z0+L) + int G) * gain, psi0c <- state
//   mode 2: out <- psi_M (FP64, no step 7)
//
// Run-time checks (text before the MPA steps: psi^{(n)} are Picard iterates
// that converge when L << z_nl).  Every level also measures its Picard
// increment at node M, Delta^{(n+1)} = psi^{(n+1)}_M - psi^{(n)}_M =
// i (D^{(n+1)} - D^{(n)}) with D the trapezoid sum of Eq. (6) at node M
// (D^{(0)} = 0), relative to |psi^{(n+1)}_M|:
//   rel_n = ||Delta^{(n+1)}|| / ||psi^{(n+1)}_M||   (sums over all frequencies).
// The last block of a link to finish (atomic ticket, no waiting) compares
// rel_n with rel_{n-1}: an increment that does not shrink, while above the
// rounding floor of the working precision, sets bit 1 of the error word
// (MPA_ERR_DIVERGED); a non-finite interval result sets bit 0.
// ERR_TIMEOUT (bit 2): a bounded wait of a persistent kernel ran out.
enum { ERR_NONFINITE = 1u, ERR_DIVERGED = 2u, ERR_TIMEOUT = 4u };
struct ConvState {
    double acc_d, acc_p;  // this level: sum |Delta|^2, sum |psi_M|^2
    double prev_rel;      // rel of the previous level of this interval
    double worst;         // largest rel_n / rel_{n-1} seen (contraction factor)
    unsigned int count;   // blocks of this level finished
    unsigned int pad;
};
// Device words of one group of links: the error word (bits above), one
// ConvState per link and D at node M per link (N complex64 each).
struct Monitor {
    unsigned int* err;
    ConvState* conv;
    float2* dprev;
    long long spin_limit;  // polls of each bounded wait of a persistent kernel
    DbgRange dbg;          // the debug build's checked range (the workspace)
};

// Natural index k = k1 + N1 k2 of position i of a node spectrum held in the
// tile layout of the staged column pass: column blocks of G = 2^logG columns,
// each G x N2 (N2 = 2^logL) contiguous, element (k2, k1 mod G) of block
// k1 / G at (k1 / G) G N2 + k2 G + k1 mod G.
__host__ __device__ __forceinline__ long long tile_to_natural(long long i, int logG, int logL, long long N) {
    const long long tb = i >> (logG + logL), rem = i & ((1ll << (logG + logL)) - 1);
    const long long k2 = rem >> logG, k1 = (tb << logG) + (rem & ((1ll << logG) - 1));
    return k1 + k2 * (N >> logL);
}

template <typename T> struct ScanParams {
    cx<T>* psi;          // link l's node j at psi + (l (M+1) + j) N
    long long N;
    int M;
    const cx<T>* psi0c;  // psi_0 in the working precision, link l at + l N
    double2* state;      // FP64 psi_0 in, A_hat(z0+L) out (mode 1), link l at + l N
    cx<T>* psi0c_out;    // mode 1: working-precision copy of the new state
    double2* out;        // mode 2
    int mode;
    const NodeC* nodes;  // node j of link l: nodes[loff[l] + j]
    const ScanNode* scn; // phases, FP32: the scan's constants, indexed as nodes
    bool phases;         // psi holds F_j and receives A_hat_j (the scan applies the phases)
    const int* loff;
    const double* gain;  // amplifier gain at the interval end, per link
    unsigned int* err;
    // Picard increment check (skipped when conv is null): level n of n_iter
    ConvState* conv;     // per link
    float2* dprev;       // D^{(n)} at node M, link l at + l N (written unless last level)
    int level, n_iter;
    double floor_rel;    // increments below this relative size are rounding, not divergence
    // tile_logG > 0: psi and dprev hold node spectra in the tile layout of the
    // staged column pass (G = 2^tile_logG columns of N2 = 2^tile_logL rows,
    // N1 = N / N2 columns); psi0c, state and out stay in natural order
    int tile_logG, tile_logL;
    DbgRange dbg;  // checked range of the debug build
};

// One thread adds a block's sums to a link's accumulators; the last of the
// level's nblk blocks closes the level (comparison with the previous one, reset).
__device__ __forceinline__ void conv_level(ConvState* cs, unsigned int* err, double sd, double sp, int level,
                                           int last_level, double floor_rel, unsigned nblk) {
    atomicAdd(&cs->acc_d, sd);
    atomicAdd(&cs->acc_p, sp);
    __threadfence();
    if (atomicAdd(&cs->count, 1u) != nblk - 1) return;
    __threadfence();
    volatile ConvState* v = cs;
    const double ad = v->acc_d, ap = v->acc_p;
    const double rel = ap > 0.0 ? sqrt(ad / ap) : 0.0;
    if (level > 0) {
        const double q = v->prev_rel > 0.0 ? rel / v->prev_rel : (rel > 0.0 ? 1e300 : 0.0);
        if (q > v->worst) v->worst = q;
        if (!(rel < v->prev_rel) && rel > floor_rel) atomicOr(err, ERR_DIVERGED);
    }
    v->prev_rel = level == last_level ? 0.0 : rel;
    v->acc_d = 0.0;
    v->acc_p = 0.0;
    v->count = 0u;
}

// The block's sums of d2 and p2 (every thread of the block calls) into link
// l's accumulators.
__device__ __forceinline__ void conv_close(ConvState* cs, unsigned int* err, double d2, double p2, int level,
                                           int last_level, double floor_rel, unsigned nblk) {
    __shared__ double red[2][32];  // one entry per warp (up to 1024 threads)
    // warp sums, then the block's warp sums by thread 0
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        d2 += __shfl_xor_sync(0xffffffffu, d2, o);
        p2 += __shfl_xor_sync(0xffffffffu, p2, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[0][w] = d2;
        red[1][w] = p2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double sd = 0.0, sp = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            sd += red[0][i];
            sp += red[1][i];
        }
        conv_level(cs, err, sd, sp, level, last_level, floor_rel, nblk);
    }
}

// What follows the sums at one frequency (position i, natural index k) of
// link l, D = (sx, sy) being the trapezoid sum of Eq. (6) at node M.
// The frequency's terms of the Picard increment check (D is kept for the
// next level):
template <typename T, bool CG>
__device__ __forceinline__ void scan_increment(const ScanParams<T>& p, int l, long long i, cx<T> p0, double sx, double sy,
                                               double& d2, double& p2) {
    const long long lo = (long long)l * p.N;
    // Picard increment at node M against the previous level's D
    double dx = sx, dy = sy;
    if (p.level > 0) {
        const float2 d0 = MPA_DBG_OK(p.dbg, p.dprev + lo + i, sizeof(float2)) ? ldx<CG>(p.dprev + lo + i)
                                                                             : make_float2(0.f, 0.f);
        dx -= (double)d0.x;
        dy -= (double)d0.y;
    }
    if (p.level < p.n_iter - 1 && MPA_DBG_OK(p.dbg, p.dprev + lo + i, sizeof(float2)))
        p.dprev[lo + i] = make_float2((float)sx, (float)sy);
    const double px = (double)p0.x - sy, py = (double)p0.y + sx;
    d2 += dx * dx + dy * dy;
    p2 += px * px + py * py;
}
// The check's sums of a block.  BLOCK: every thread of the block calls, the
// sums go through a block reduction; else one whole warp of the block calls,
// and its sums are the block's.
template <typename T, bool BLOCK>
__device__ __forceinline__ void scan_check(const ScanParams<T>& p, int l, double d2, double p2, unsigned nblk) {
    if constexpr (BLOCK) {
        conv_close(p.conv + l, p.err, d2, p2, p.level, p.n_iter - 1, p.floor_rel, nblk);
    } else {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            d2 += __shfl_xor_sync(0xffffffffu, d2, o);
            p2 += __shfl_xor_sync(0xffffffffu, p2, o);
        }
        if ((threadIdx.x & 31) == 0) conv_level(p.conv + l, p.err, d2, p2, p.level, p.n_iter - 1, p.floor_rel, nblk);
    }
}
// At the last level, step 7 (mode 1) or psi_M (mode 2):
template <typename T, bool CG>
__device__ __forceinline__ void scan_finish(const ScanParams<T>& p, int l, long long k, double sx, double sy) {
    typedef cx<T> C;
    const long long lo = (long long)l * p.N;
    const double2 s0 = MPA_DBG_OK(p.dbg, p.state + lo + k, sizeof(double2)) ? ldx<CG>(p.state + lo + k)
                                                                          : make_double2(0.0, 0.0);
    const double2 psiM = make_double2(s0.x - sy, s0.y + sx);
    if (p.mode == 2) {
        p.out[lo + k] = psiM;  // the caller's buffer (mpa_interval), outside the workspace
        return;
    }
    // step 7 and the lumped gain
    NodeC nodeM{};
    if (MPA_DBG_OK(p.dbg, p.loff + l, sizeof(int)) && MPA_DBG_OK(p.dbg, p.nodes + p.loff[l] + p.M, sizeof(NodeC)))
        nodeM = p.nodes[p.loff[l] + p.M];
    const double2 ph = expi_turns<double>(phase_q64(signed_k(k, p.N), nodeM));
    const double g = nodeM.pre * (MPA_DBG_OK(p.dbg, p.gain + l, sizeof(double)) ? p.gain[l] : 0.0);
    const double2 a = make_double2(g * (psiM.x * ph.x - psiM.y * ph.y), g * (psiM.x * ph.y + psiM.y * ph.x));
    if (MPA_DBG_OK(p.dbg, p.state + lo + k, sizeof(double2))) p.state[lo + k] = a;
    if (MPA_DBG_OK(p.dbg, p.psi0c_out + lo + k, sizeof(C))) p.psi0c_out[lo + k] = mkc((T)a.x, (T)a.y);
    if (!(isfinite(a.x) && isfinite(a.y))) atomicOr(p.err, ERR_NONFINITE);
}

// All of it for one frequency, and for the pair k, k + 1 at positions i, i + 1.
template <typename T, bool CG, bool BLOCK>
__device__ __forceinline__ void scan_node_m(const ScanParams<T>& p, int l, long long i, long long k, cx<T> p0, double sx,
                                            double sy, unsigned nblk) {
    if (p.conv) {
        double d2 = 0.0, p2 = 0.0;
        scan_increment<T, CG>(p, l, i, p0, sx, sy, d2, p2);
        scan_check<T, BLOCK>(p, l, d2, p2, nblk);
    }
    if (p.mode != 0) scan_finish<T, CG>(p, l, k, sx, sy);
}
template <bool BLOCK>
__device__ __forceinline__ void scan_pair_m(const ScanParams<float>& p, int l, long long i, long long k, float2 pa, float2 pb,
                                            double ax, double ay, double bx, double by, unsigned nblk) {
    if (p.conv) {
        double d2 = 0.0, p2 = 0.0;
        scan_increment<float, false>(p, l, i, pa, ax, ay, d2, p2);
        scan_increment<float, false>(p, l, i + 1, pb, bx, by, d2, p2);
        scan_check<float, BLOCK>(p, l, d2, p2, nblk);
    }
    if (p.mode != 0) {
        scan_finish<float, false>(p, l, k, ax, ay);
        scan_finish<float, false>(p, l, k + 1, bx, by);
    }
}

// s += v, Kahan-compensated in FP32 (c carries the lost low-order part; the
// float2 sums and differences are packed instructions), plain in FP64.
template <class C> __device__ __forceinline__ void scan_add(C& s, C& c, C v) {
    if constexpr (sizeof(C) == 8) {
        const C y = csub(v, c), t = cadd(s, y);
        c = csub(csub(t, s), y);
        s = t;
    } else {
        s = cadd(s, v);
    }
}
// s - c + v / 2
template <class C> __device__ __forceinline__ C scan_half(C s, C c, C v) {
    if constexpr (sizeof(C) == 8) return cadd(csub(s, c), cscale(v, 0.5f));
    else return mkc(s.x + 0.5 * v.x, s.y + 0.5 * v.y);
}

// 16-byte global -> shared copy through L2 (cp.async.cg) and its commit /
// wait groups
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait_group() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Frequency k of link l (one thread each; a block of consecutive
// frequencies, nblk blocks per link).  N is a multiple of the block size (a
// power of two >= 256), so every thread has a frequency and takes part in
// the block reduction of the increment check.
// PH (ScanParams::phases; FP64 plans): psi holds F_j and receives A_hat_j,
// every phase from its node's own constants; else (also the persistent batch
// kernel) it holds V_j and receives psi_j.  Nodes are loaded 8 ahead.
template <typename T, bool CG, bool PH>
__device__ __forceinline__ void scan_freq(const ScanParams<T>& p, int l, long long i, unsigned nblk) {
    typedef cx<T> C;
    const long long lo = (long long)l * p.N;
    // i: position in the node buffers; k: the frequency there (natural order)
    cx<T>* psi = p.psi + lo * (p.M + 1) + i;
    const long long k = p.tile_logG > 0 ? tile_to_natural(i, p.tile_logG, p.tile_logL, p.N) : i;
    const long long kk = signed_k(k, p.N);
    const C zero = mkc(T(0), T(0));
    const C v0 = MPA_DBG_OK(p.dbg, psi, sizeof(C)) ? ldx<CG>(psi) : zero;
    const C p0 = MPA_DBG_OK(p.dbg, p.psi0c + lo + k, sizeof(C)) ? ldx<CG>(p.psi0c + lo + k) : zero;
    const NodeC* nodes = nullptr;
    auto consts = [&](int j) {
        NodeC nc{};
        if (MPA_DBG_OK(p.dbg, nodes + j, sizeof(NodeC))) nc = nodes[j];
        return nc;
    };
    C vl = v0;
    if constexpr (PH) {
        if (MPA_DBG_OK(p.dbg, p.loff + l, sizeof(int))) nodes = p.nodes + p.loff[l];
        vl = cscale(v0, (T)consts(0).post);  // phase 0 and factor 1: V_0 = sigma_0 dz F_0
    }
    C r = cscale(vl, T(0.5)), c = zero;
    // node j: psi^{(n+1)}_j = psi_0 + i (R + V_j/2), then R += V_j
    auto node = [&](int j, C v) {
        C ph;
        vl = v;
        if constexpr (PH) {
            const NodeC nc = consts(j);
            ph = expi_turns<T>(phase_q64(kk, nc));
            vl = cscale(cmul(v, cconj(ph)), (T)nc.post);
            ph = cscale(ph, (T)nc.pre);
        }
        if (p.mode == 0) {
            const C h = scan_half(r, c, vl);
            C o = mkc(p0.x - h.y, p0.y + h.x);
            if constexpr (PH) o = cmul(o, ph);
            if (MPA_DBG_OK(p.dbg, psi + (long long)j * p.N, sizeof(C))) psi[(long long)j * p.N] = o;
        }
        scan_add(r, c, vl);
    };
    // the loads never touch a node the loop has written (they run ahead)
    constexpr int U = 8;
    C nxt[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
        nxt[u] = (1 + u <= p.M && MPA_DBG_OK(p.dbg, psi + (long long)(1 + u) * p.N, sizeof(C)))
                     ? ldx<CG>(psi + (long long)(1 + u) * p.N)
                     : zero;
    for (int jb = 1; jb <= p.M; jb += U) {
        C cur[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            cur[u] = nxt[u];
            const int jn = jb + U + u;
            nxt[u] = (jn <= p.M && MPA_DBG_OK(p.dbg, psi + (long long)jn * p.N, sizeof(C)))
                         ? ldx<CG>(psi + (long long)jn * p.N)
                         : zero;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int j = jb + u;
            if (j > p.M) break;
            node(j, cur[u]);
        }
    }
    // D = R_M - V_M/2 at node M in FP64 (psi_M = psi_0 + i D)
    const double sx = ((double)r.x - (double)c.x) - 0.5 * (double)vl.x;
    const double sy = ((double)r.y - (double)c.y) - 0.5 * (double)vl.y;
    if constexpr (!CG) pdl_go();
    scan_node_m<T, CG, true>(p, l, i, k, p0, sx, sy, nblk);
}

template <typename T, bool PH> __global__ void __launch_bounds__(256) scan_kernel(const ScanParams<T> p) {
    pdl_wait();
    scan_freq<T, false, PH>(p, blockIdx.y, (long long)blockIdx.x * blockDim.x + threadIdx.x, gridDim.x);
}

// ---- FP32: two neighbouring frequencies a thread.
// The phases at a pair of frequencies k, k + 1, walked in node order: one
// evaluation of the pair a node (packed), the phases advanced by their steps
// (64-bit adds; a step is evaluated again only where the fiber segment
// changes).
struct PairWalk {
    const ScanNode* sn;
    const DbgRange& dbg;
    long long ka, kb;
    unsigned long long ta = 0, tb = 0, da = 0, db = 0;
    int fresh = 0;  // the next node whose step is not the current one
    __device__ __forceinline__ PairWalk(const ScanParams<float>& p, int l, long long k)
        : sn(p.scn + (MPA_DBG_OK(p.dbg, p.loff + l, sizeof(int)) ? p.loff[l] : 0)), dbg(p.dbg), ka(signed_k(k, p.N)),
          kb(signed_k(k + 1, p.N)) {}
    // the step from node j on
    __device__ __forceinline__ void step(int j) {
        fresh = INT_MAX;
        if (!MPA_DBG_OK(dbg, sn + j, sizeof(ScanNode))) return;
        const ScanNode& s = sn[j];
        da = phase_q64(ka, s.da_hi, s.da_lo, s.db_hi, s.db_lo);
        db = phase_q64(kb, s.da_hi, s.da_lo, s.db_hi, s.db_lo);
        fresh = s.next;
    }
    // (pre, pre, post, post) of node j
    __device__ __forceinline__ float4 consts(int j) const {
        const float4* a = reinterpret_cast<const float4*>(sn[j].pre);
        return MPA_DBG_OK(dbg, a, 16) ? __ldg(a) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    // exp(i beta_j) at both frequencies, then on to node j + 1
    __device__ __forceinline__ void next(float2& ea, float2& eb) {
        expi_turns_poly2(ta, tb, ea, eb);
        ta += da;
        tb += db;
    }
};
__device__ __forceinline__ float2 f4a(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 f4b(float4 v) { return make_float2(v.z, v.w); }
__device__ __forceinline__ float4 f4(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

// The FP32 scan: a thread walks all nodes of two frequencies; its nodes
// travel SCAN_S ahead through its own shared-memory slots by 16-byte
// cp.async, so the bytes in flight do not cost registers.  STORE: mode 0.
// 16 slots and five blocks an SM: 266 us a level at 2^20 x 126 nodes (the
// scan without phases 261 us: the phases hide behind HBM), 126 us at 2^16 x
// 801; 8 slots and eight blocks 270 and 140 us.
constexpr int SCAN_S = 16, SCAN_NT = 128;
template <bool STORE> __global__ void __launch_bounds__(SCAN_NT, 5) scan_pair_kernel(const ScanParams<float> p) {
    __shared__ float4 ring[SCAN_S * SCAN_NT];
    __shared__ float4 cst[SCAN_NT];  // PairWalk::consts of the nodes at hand
    pdl_wait();
    const int l = blockIdx.y;
    const long long i = 2 * ((long long)blockIdx.x * SCAN_NT + threadIdx.x);
    const long long lo = (long long)l * p.N, N2 = p.N >> 1;  // N2: float4 distance of nodes
    float4* psi = reinterpret_cast<float4*>(p.psi + lo * (p.M + 1) + i);
    // a pair shares a row of the tile layout, so its frequencies are neighbours there too
    const long long k = p.tile_logG > 0 ? tile_to_natural(i, p.tile_logG, p.tile_logL, p.N) : i;
    const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
    float4* mine = ring + threadIdx.x;
    const float4* ld = psi;
#pragma unroll
    for (int u = 0; u < SCAN_S; ++u) {
        ld += N2;
        if (1 + u <= p.M && MPA_DBG_OK(p.dbg, ld, 16)) cp_async16(mine + u * SCAN_NT, ld);
        cp_async_commit();
    }
    const float4 v0 = MPA_DBG_OK(p.dbg, psi, 16) ? *psi : zero;
    const float4* p0p = reinterpret_cast<const float4*>(p.psi0c + lo + k);
    const float4 p0 = MPA_DBG_OK(p.dbg, p0p, 16) ? *p0p : zero;
    const float2 pa = f4a(p0), pb = f4b(p0);
    PairWalk walk(p, l, k);
    // node 0: phase 0 and factor 1, V_0 = sigma_0 dz F_0
    const float2 post0 = f4b(walk.consts(0));
    float2 va = mul2(f4a(v0), post0), vb = mul2(f4b(v0), post0);
    const float2 half = make_float2(0.5f, 0.5f);
    float2 ra = mul2(va, half), rb = mul2(vb, half), ca = make_float2(0.f, 0.f), cb = ca;
    walk.step(0);
    walk.ta = walk.da;  // node 1
    walk.tb = walk.db;
    if (walk.fresh == 1) walk.step(1);
    float2 na, nb;
    walk.next(na, nb);
    float4* st = psi;
    int slot = 0;
    for (int jb = 1; jb <= p.M; jb += SCAN_NT) {
        // the factors of the next SCAN_NT nodes
        const int je = p.M + 1 - jb < SCAN_NT ? p.M + 1 : jb + SCAN_NT;
        __syncthreads();
        if (jb + (int)threadIdx.x < je) cst[threadIdx.x] = walk.consts(jb + (int)threadIdx.x);
        __syncthreads();
        for (int j = jb; j < je;) {
            // the loop takes the step from node j + 1 on: up to the node before the next change
            if (j + 1 == walk.fresh) walk.step(j + 1);
            // (any other value of fresh takes the rest of the nodes: the loop always advances)
            const int end = walk.fresh > j + 1 && walk.fresh <= je ? walk.fresh - 1 : je;
#pragma unroll 2
            for (; j < end; ++j) {
                const float4 w = cst[j - jb];
                const float2 ea = na, eb = nb;
                walk.next(na, nb);  // node j + 1's phases, beside node j's sums
                cp_async_wait_group<SCAN_S - 1>();  // node j's copy has landed
                float4* sl = mine + slot * SCAN_NT;
                const float4 v = *sl;
                slot = (slot + 1) & (SCAN_S - 1);
                ld += N2;
                st += N2;
                va = mul2(cmul(f4a(v), cconj(ea)), f4b(w));
                vb = mul2(cmul(f4b(v), cconj(eb)), f4b(w));
                if constexpr (STORE) {
                    // psi^{(n+1)}_j = psi_0 + i (R + V_j/2), stored with its phase and loss
                    const float2 ha = fma2(va, half, csub(ra, ca)), hb = fma2(vb, half, csub(rb, cb));
                    const float2 oa = cmul(make_float2(pa.x - ha.y, pa.y + ha.x), mul2(ea, f4a(w)));
                    const float2 ob = cmul(make_float2(pb.x - hb.y, pb.y + hb.x), mul2(eb, f4a(w)));
                    if (MPA_DBG_OK(p.dbg, st, 16)) *st = f4(oa, ob);
                }
                scan_add(ra, ca, va);
                scan_add(rb, cb, vb);
                // the slot's value is consumed: refill it with node j + SCAN_S
                if (j + SCAN_S <= p.M && MPA_DBG_OK(p.dbg, ld, 16)) cp_async16(sl, ld);
                cp_async_commit();
            }
        }
    }
    cp_async_wait_group<0>();
    pdl_go();
    // D = R_M - V_M/2 at node M in FP64 (psi_M = psi_0 + i D)
    scan_pair_m<true>(p, l, i, k, pa, pb, ((double)ra.x - (double)ca.x) - 0.5 * (double)va.x,
                      ((double)ra.y - (double)ca.y) - 0.5 * (double)va.y, ((double)rb.x - (double)cb.x) - 0.5 * (double)vb.x,
                      ((double)rb.y - (double)cb.y) - 0.5 * (double)vb.y, gridDim.x);
}

// The scan with the nodes of a frequency split over the block: 32 frequencies
// (lanes) x SCS_W warps, warp w taking a run of up to SCS_C consecutive nodes
// of each panel of nodes.  A thread loads its run into registers at once and
// sums it; the runs' sums are combined through shared memory (compensated in
// FP32 like the sums themselves), and the thread adds its exclusive prefix to
// the run's partial sums.  A thread per frequency leaves a short link with few
// warps that each walk all M nodes one after another (N = 2^12: 16 blocks on
// 152 SMs, bound by L2 latency); here every node of a panel is in flight at
// once: FP32 21.3 -> 13.2 us at 2^12 x 143 nodes, 21.0 -> 14.2 at 2^13 x 143,
// 65.6 -> 22.2 at 2^12 x 801, 65.9 -> 27.0 at 2^13 x 801.  Eight warps at 64
// registers (FP32 spills 48 bytes): four blocks an SM, whose load, sum and store
// phases overlap (at 2^14 x 801, which takes the scan with phases since, 43 us;
// 16 warps at 64 registers 52, at 101 registers 66).
constexpr int SCS_W = 8;
template <typename T>
__global__ void __launch_bounds__(32 * SCS_W, sizeof(T) == 4 ? 4 : 2) scan_split_kernel(const ScanParams<T> p) {
    typedef cx<T> C;
    constexpr bool F32 = sizeof(T) == 4;
    constexpr int SCS_C = F32 ? 16 : 8;         // nodes a thread holds
    __shared__ C ps[SCS_W][32], pc[SCS_W][32];  // the runs' sums and compensations
    pdl_wait();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, l = blockIdx.y;
    const long long i = (long long)blockIdx.x * 32 + lane;
    const long long lo = (long long)l * p.N;
    C* psi = p.psi + lo * (p.M + 1) + i;
    const long long k = p.tile_logG > 0 ? tile_to_natural(i, p.tile_logG, p.tile_logL, p.N) : i;
    const C zero = mkc(T(0), T(0));
    const C v0 = MPA_DBG_OK(p.dbg, psi, sizeof(C)) ? *psi : zero;
    const C p0 = MPA_DBG_OK(p.dbg, p.psi0c + lo + k, sizeof(C)) ? p.psi0c[lo + k] : zero;
    // equal runs: as few panels as the registers allow, nodes spread evenly over them
    const int panels = (p.M + SCS_W * SCS_C - 1) / (SCS_W * SCS_C);
    const int run = (p.M + SCS_W * panels - 1) / (SCS_W * panels);
    C r = mkc(T(0.5) * v0.x, T(0.5) * v0.y), c = zero;  // sum before the panel and its compensation
    for (int jb = 1; jb <= p.M; jb += SCS_W * run) {
        const int j0 = jb + w * run;
        const int n = p.M + 1 - j0 < run ? p.M + 1 - j0 : run;  // nodes of this thread's run (<= 0: none)
        C* a = psi + (long long)j0 * p.N;
        C v[SCS_C];
#pragma unroll
        for (int u = 0; u < SCS_C; ++u)
            v[u] = u < n && MPA_DBG_OK(p.dbg, a + (long long)u * p.N, sizeof(C)) ? a[(long long)u * p.N] : zero;
        // v[u] <- (sum of the run before node u) + V_u / 2
        C s = zero, sc = zero, vl = zero;
#pragma unroll
        for (int u = 0; u < SCS_C; ++u) {
            const C x = v[u];
            if (u < n) vl = x;
            v[u] = mkc((F32 ? s.x - sc.x : s.x) + T(0.5) * x.x, (F32 ? s.y - sc.y : s.y) + T(0.5) * x.y);
            if constexpr (F32) {
                kahan_add(s.x, sc.x, x.x);
                kahan_add(s.y, sc.y, x.y);
            } else {
                s.x += x.x;
                s.y += x.y;
            }
        }
        if (jb > 1) __syncthreads();  // the previous panel's sums have been read
        if (jb + SCS_W * run > p.M) pdl_go();
        ps[w][lane] = s;
        if constexpr (F32) pc[w][lane] = sc;
        __syncthreads();
        C mr = r, mc = c;  // sum before this thread's run
#pragma unroll
        for (int q = 0; q < SCS_W; ++q) {
            if (q == w) {
                mr = r;
                mc = c;
            }
            const C t = ps[q][lane];
            if constexpr (F32) {
                const C tc = pc[q][lane];
                kahan_add(r.x, c.x, t.x);
                kahan_add(r.y, c.y, t.y);
                c.x += tc.x;
                c.y += tc.y;
            } else {
                r.x += t.x;
                r.y += t.y;
            }
        }
        if (p.mode == 0) {
            const C b = F32 ? mkc(mr.x - mc.x, mr.y - mc.y) : mr;
#pragma unroll
            for (int u = 0; u < SCS_C; ++u)
                if (u < n && MPA_DBG_OK(p.dbg, a + (long long)u * p.N, sizeof(C)))
                    a[(long long)u * p.N] = mkc(p0.x - (b.y + v[u].y), p0.y + (b.x + v[u].x));
        }
        if (n > 0 && j0 + n == p.M + 1) {  // the warp of node M
            // D = R_M - V_M/2 at node M in FP64, R_M = the sum before the run + the run
            double sx = (double)mr.x + (double)s.x, sy = (double)mr.y + (double)s.y;
            if constexpr (F32) {
                sx -= (double)mc.x + (double)sc.x;
                sy -= (double)mc.y + (double)sc.y;
            }
            scan_node_m<T, false, false>(p, l, i, k, p0, sx - 0.5 * (double)vl.x, sy - 0.5 * (double)vl.y, gridDim.x);
        }
    }
}

// out[c][r] = in[r][c] for an R x Cc matrix (32 x 32 tiles).
template <typename T>
__global__ void __launch_bounds__(256) transpose_kernel(const cx<T>* __restrict__ in, cx<T>* __restrict__ out,
                                                         long long R, long long Cc) {
    __shared__ cx<T> t[32][33];
    pdl_go();
    pdl_wait();
    const long long r0 = (long long)blockIdx.y * 32, c0 = (long long)blockIdx.x * 32;
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long r = r0 + y, c = c0 + threadIdx.x;
        if (r < R && c < Cc) t[y][threadIdx.x] = in[r * Cc + c];
    }
    __syncthreads();
    for (int y = threadIdx.y; y < 32; y += 8) {
        const long long c = c0 + y, r = r0 + threadIdx.x;
        if (r < R && c < Cc) out[c * R + r] = t[threadIdx.x][y];
    }
}

// Precision conversions between the FP64 state and working buffers.
template <typename T>
__global__ void __launch_bounds__(256) to_state_kernel(const cx<T>* in, double2* state, cx<T>* copy, long long N) {
    pdl_go();
    pdl_wait();
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    const cx<T> v = in[k];
    state[k] = make_double2((double)v.x, (double)v.y);
    if (copy) copy[k] = v;
}
template <typename T>
__global__ void __launch_bounds__(256) from_state_kernel(const double2* state, cx<T>* out, long long N) {
    pdl_go();
    pdl_wait();
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= N) return;
    const double2 v = state[k];
    out[k] = mkc((T)v.x, (T)v.y);
}

}  // namespace mpa
