// Column-pass launchers, double.
#include "launch.h"

namespace mpa {

template <int L, int MODE, int F = 0>
static cudaError_t kc_one(const KCParams<double>& pin, cudaStream_t st) {
    if (const cudaError_t eg = launch_gate()) return eg;
    // callers that leave the link fields unset launch one run of nodes
    KCParams<double> p = pin;
    if (p.npl <= 0) p.npl = (int)(p.ncols >> p.logN1) > 0 ? (int)(p.ncols >> p.logN1) : 1;
    typedef KCGeom<double, L, F> Gm;
    static AttrOnce once;
    const cudaError_t ea = attrs_once(once, [] {
        cudaError_t e = cudaFuncSetAttribute(kc_kernel<double, L, MODE, F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)Gm::smem_bytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kc_kernel<double, L, MODE, F>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        return cudaSuccess;
    });
    if (ea != cudaSuccess) return ea;
    const long long nblk = (p.ncols + Gm::G - 1) / Gm::G;
    if (nblk <= 0) return cudaSuccess;
    bool early;
    if constexpr (F == 0) {
        int sms = 0;
        const cudaError_t es = sm_count(&sms);
        if (es != cudaSuccess) return es;
        early = pdl_level64(pair_fits(Gm::smem_bytes), nblk, sms);
    } else {
        early = pdl_field<double>(p.N, MODE == KC_FWDF || MODE == KC_FWD_T || MODE == KC_INV || MODE == KC_INV_T);
    }
    const bool prof = g_prof_on.load(std::memory_order_relaxed);
    if (prof) prof_begin(st);
    const cudaError_t el =
        launch_pdl(early, kc_kernel<double, L, MODE, F>, (unsigned)nblk, Gm::NT, Gm::smem_bytes, st, p);
    if (prof) {
        // algorithmic bytes: every tile element read once and written once
        // (a shared source, src_stride == 0, is read once for all nodes)
        const double cs = (double)sizeof(cx<double>), tile = (double)p.ncols * L;
        const double rd = p.src_stride == 0 ? (double)p.ncols / p.npl * L : tile;
        prof_end(prof_kc_kind(MODE, p.err != nullptr), st, (rd + tile) * cs);
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return el;
}

template <int L, int MODE> static cudaError_t kc_field(const KCParams<double>& p, cudaStream_t st) {
    return field_tiles<double>(L, p.ncols * L) == 1 ? kc_one<L, MODE, 1>(p, st) : kc_one<L, MODE, 2>(p, st);
}

template <int L>
static cudaError_t kc_mode(int mode, const KCParams<double>& p, cudaStream_t st) {
    // passes of the MPA levels (error word) are many nodes: large tiles
    switch (mode) {
        case KC_MPA_PRE: return kc_one<L, KC_MPA_PRE>(p, st);
        case KC_MPA_POST: return kc_one<L, KC_MPA_POST>(p, st);
        case KC_SS_STEP: return kc_field<L, KC_SS_STEP>(p, st);
        case KC_FWD: return p.err ? kc_one<L, KC_FWD>(p, st) : kc_field<L, KC_FWD>(p, st);
        case KC_INV: return p.err ? kc_one<L, KC_INV>(p, st) : kc_field<L, KC_INV>(p, st);
        case KC_FWDF: return kc_field<L, KC_FWDF>(p, st);
        case KC_FWD_T: return kc_field<L, KC_FWD_T>(p, st);
        case KC_INV_T: return kc_field<L, KC_INV_T>(p, st);
    }
    return cudaErrorInvalidValue;
}

template <>
cudaError_t kc_launch<double>(int mode, int logL, const KCParams<double>& p, cudaStream_t st) {
    switch (logL) {
        case 4: return kc_mode<16>(mode, p, st);
        case 5: return kc_mode<32>(mode, p, st);
        case 6: return kc_mode<64>(mode, p, st);
        case 7: return kc_mode<128>(mode, p, st);
        case 8: return kc_mode<256>(mode, p, st);
        case 9: return kc_mode<512>(mode, p, st);
        case 10: return kc_mode<1024>(mode, p, st);
        case 11: return kc_mode<2048>(mode, p, st);
    }
    return cudaErrorInvalidValue;
}

template <>
long long kc_blocks<double>(int logL, long long ncols) {
    switch (logL) {
        case 4: return (ncols + KCGeom<double, 16>::G - 1) / KCGeom<double, 16>::G;
        case 5: return (ncols + KCGeom<double, 32>::G - 1) / KCGeom<double, 32>::G;
        case 6: return (ncols + KCGeom<double, 64>::G - 1) / KCGeom<double, 64>::G;
        case 7: return (ncols + KCGeom<double, 128>::G - 1) / KCGeom<double, 128>::G;
        case 8: return (ncols + KCGeom<double, 256>::G - 1) / KCGeom<double, 256>::G;
        case 9: return (ncols + KCGeom<double, 512>::G - 1) / KCGeom<double, 512>::G;
        case 10: return (ncols + KCGeom<double, 1024>::G - 1) / KCGeom<double, 1024>::G;
        case 11: return (ncols + KCGeom<double, 2048>::G - 1) / KCGeom<double, 2048>::G;
    }
    return -1;
}

}  // namespace mpa
