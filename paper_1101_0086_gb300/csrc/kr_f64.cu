// Row-pass launchers, double.
#include "launch.h"

namespace mpa {

template <int L, int MODE, int F = 0>
static cudaError_t kr_one(const KRParams<double>& p, cudaStream_t st) {
    if (const cudaError_t eg = launch_gate()) return eg;
    typedef KRGeom<double, L, F> Gm;
    static AttrOnce once;
    const cudaError_t ea = attrs_once(once, [] {
        cudaError_t e = cudaFuncSetAttribute(kr_kernel<double, L, MODE, F>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)Gm::smem_bytes);
        if (e != cudaSuccess) return e;
        e = cudaFuncSetAttribute(kr_kernel<double, L, MODE, F>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        if (e != cudaSuccess) return e;
        return cudaSuccess;
    });
    if (ea != cudaSuccess) return ea;
    const long long nblk = (p.nrows + Gm::G - 1) / Gm::G;
    if (nblk <= 0) return cudaSuccess;
    bool early;
    if constexpr (F == 0) {
        int sms = 0;
        const cudaError_t es = sm_count(&sms);
        if (es != cudaSuccess) return es;
        early = pdl_level64(pair_fits(Gm::smem_bytes), nblk, sms);
    } else {
        early = pdl_field<double>(p.N);
    }
    const bool prof = g_prof_on.load(std::memory_order_relaxed);
    if (prof) prof_begin(st);
    const cudaError_t el =
        launch_pdl(early, kr_kernel<double, L, MODE, F>, (unsigned)nblk, Gm::NT, Gm::smem_bytes, st, p);
    if (prof) prof_end(prof_kr_kind(MODE), st, 2.0 * (double)p.nrows * L * sizeof(cx<double>));
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return el;
}

template <int L, int MODE> static cudaError_t kr_field(const KRParams<double>& p, cudaStream_t st) {
    if constexpr (field_tiles<double>(L, 0) == 0) return kr_one<L, MODE>(p, st);
    else return field_tiles<double>(L, p.nrows * L) == 1 ? kr_one<L, MODE, 1>(p, st) : kr_one<L, MODE, 2>(p, st);
}

template <int L>
static cudaError_t kr_mode(int mode, const KRParams<double>& p, cudaStream_t st) {
    switch (mode) {
        case KR_MPA: return kr_one<L, KR_MPA>(p, st);
        case KR_SS: return kr_field<L, KR_SS>(p, st);
        case KR_FWD: return kr_field<L, KR_FWD>(p, st);
        case KR_INV: return kr_field<L, KR_INV>(p, st);
    }
    return cudaErrorInvalidValue;
}

template <>
cudaError_t kr_launch<double>(int mode, int logL, const KRParams<double>& p, cudaStream_t st) {
    switch (logL) {
        case 4: return kr_mode<16>(mode, p, st);
        case 5: return kr_mode<32>(mode, p, st);
        case 6: return kr_mode<64>(mode, p, st);
        case 7: return kr_mode<128>(mode, p, st);
        case 8: return kr_mode<256>(mode, p, st);
        case 9: return kr_mode<512>(mode, p, st);
        case 10: return kr_mode<1024>(mode, p, st);
        case 11: return kr_mode<2048>(mode, p, st);
        case 12: return kr_mode<4096>(mode, p, st);
        case 13: return kr_mode<8192>(mode, p, st);
    }
    return cudaErrorInvalidValue;
}

template <>
long long kr_blocks<double>(int logL, long long nrows) {
    switch (logL) {
        case 4: return (nrows + KRGeom<double, 16>::G - 1) / KRGeom<double, 16>::G;
        case 5: return (nrows + KRGeom<double, 32>::G - 1) / KRGeom<double, 32>::G;
        case 6: return (nrows + KRGeom<double, 64>::G - 1) / KRGeom<double, 64>::G;
        case 7: return (nrows + KRGeom<double, 128>::G - 1) / KRGeom<double, 128>::G;
        case 8: return (nrows + KRGeom<double, 256>::G - 1) / KRGeom<double, 256>::G;
        case 9: return (nrows + KRGeom<double, 512>::G - 1) / KRGeom<double, 512>::G;
        case 10: return (nrows + KRGeom<double, 1024>::G - 1) / KRGeom<double, 1024>::G;
        case 11: return (nrows + KRGeom<double, 2048>::G - 1) / KRGeom<double, 2048>::G;
        case 12: return (nrows + KRGeom<double, 4096>::G - 1) / KRGeom<double, 4096>::G;
        case 13: return (nrows + KRGeom<double, 8192>::G - 1) / KRGeom<double, 8192>::G;
    }
    return -1;
}

}  // namespace mpa
