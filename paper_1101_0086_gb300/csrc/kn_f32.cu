// Launchers of the on-chip whole node transform, float.
#include "launch.h"

namespace mpa {

template <int L, bool PIN, bool POUT, int F>
static cudaError_t kn_one(const KNParams<float>& p, cudaStream_t st) {
    if (const cudaError_t eg = launch_gate()) return eg;
    typedef KNGeom<float, L, F> Gm;
    static AttrOnce once;
    const cudaError_t ea = attrs_once(once, [] {
        cudaError_t e = cudaFuncSetAttribute(kn_kernel<float, L, PIN, POUT, F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)Gm::smem_bytes);
        if (e != cudaSuccess) return e;
        return cudaFuncSetAttribute(kn_kernel<float, L, PIN, POUT, F>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    });
    if (ea != cudaSuccess) return ea;
    const long long nblk = (p.nrows + Gm::G - 1) / Gm::G;
    if (nblk <= 0) return cudaSuccess;
    const bool prof = g_prof_on.load(std::memory_order_relaxed);
    if (prof) prof_begin(st);
    const cudaError_t el =
        launch_pdl(pdl_fills(nblk), kn_kernel<float, L, PIN, POUT, F>, (unsigned)nblk, Gm::NT, Gm::smem_bytes, st, p);
    if (prof) {
        // every node read once and written once (a shared psi_0 once per link)
        const double cs = (double)sizeof(cx<float>), nodes = (double)p.nrows;
        const double rd = p.src_stride == 0 ? nodes / p.npl : nodes;
        prof_end(PK_KN, st, (rd + nodes) * L * cs);
    }
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return el;
}

// Whether a launch takes the fine tiles: up to 2^12 modes, where the large
// ones (8192 elements) would not fill the SMs twice.  Measured, us a launch,
// large / fine: 143 nodes 2^8 14.2 / 8.6, 2^10 13.3 / 10.1, 2^12 15.7 / 11.5, 2^13
// 16.4 / 17.2, 2^14 19.6 / 22.7; 801 nodes 2^11 (201 tiles) 22.6 / 18.4, 2^12
// (401 tiles) 31.7 / 32.7.
template <int L> static bool kn_fine(const KNParams<float>& p, int sms) {
    return !fills_twice((p.nrows + KNGeom<float, L>::G - 1) / KNGeom<float, L>::G, sms);
}

template <int L, bool PIN, bool POUT> static cudaError_t kn_any(const KNParams<float>& p, cudaStream_t st) {
    if constexpr (L <= 4096) {
        int sms = 0;
        const cudaError_t e = sm_count(&sms);
        if (e != cudaSuccess) return e;
        if (kn_fine<L>(p, sms)) return kn_one<L, PIN, POUT, 1>(p, st);
    }
    return kn_one<L, PIN, POUT, 0>(p, st);
}
template <int L> static cudaError_t kn_len(const KNParams<float>& p, cudaStream_t st) {
    if (p.phase_out) return p.phase_in ? kn_any<L, true, true>(p, st) : cudaErrorInvalidValue;
    return p.phase_in ? kn_any<L, true, false>(p, st) : kn_any<L, false, false>(p, st);
}

template <>
cudaError_t kn_launch<float>(int logL, const KNParams<float>& p, cudaStream_t st) {
    switch (logL) {
        case 8: return kn_len<256>(p, st);
        case 9: return kn_len<512>(p, st);
        case 10: return kn_len<1024>(p, st);
        case 11: return kn_len<2048>(p, st);
        case 12: return kn_len<4096>(p, st);
        case 13: return kn_len<8192>(p, st);
        case 14: return kn_len<16384>(p, st);
        case 15:
        case 16: return knc_launch(logL, p, st);
    }
    return cudaErrorInvalidValue;
}

}  // namespace mpa
