// Host-side check of the twiddle tables' places and contents (no GPU needed):
// - the direct table of the staged column passes (kcs.cuh) lies between the
//   two-level tables and the groups' buffers, 16-byte aligned for its 16-byte
//   reads, and holds the entries of both transforms;
// - the two-level tables with residuals and the whole tables fit the room that
//   the tiles keep for them, before the outer factors;
// - W_32 in FP32 and its residuals (w32) add up to the closed forms;
// - the split slot form (Slot) equals the padded slot at every site of the
//   passes on the fine FP64 tiles, whose padding shift is 2.
// Prints the number of checks; exits non-zero on the first failure.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "kcs.cuh"

using namespace mpa;

static long long g_checked = 0;

static void expect_true(bool ok, const char* what, int L) {
    ++g_checked;
    if (!ok) {
        std::printf("failed: %s (L = %d)\n", what, L);
        std::exit(1);
    }
}

template <int L> void staged_direct_table() {
    typedef KCSGeom<L> SG;
    const size_t C = sizeof(float2), end = SG::DT_OFF + (size_t)SG::DTN * C;
    expect_true(SG::DT_OFF % 16 == 0, "16-byte reads of the direct table", L);
    expect_true(SG::TW_OFF + (size_t)Tw<float, L>::N * C <= SG::DT_OFF && end <= SG::GRP_OFF, "between tables and groups", L);
    expect_true(SG::XF::DTN <= SG::DTN && SG::XI::DTN <= SG::DTN && SG::DTN <= 1024, "entries of both transforms", L);
    // dt_row's highest entry is the table's last: float4 (R/2 - 1) NS + NS - 1
    expect_true(SG::XI::DTN == SG::XI::NS1 * SG::XI::R1 && 2 * ((SG::XI::R1 / 2 - 1) * SG::XI::NS1 + SG::XI::NS1) <= SG::DTN,
                "reads inside the table", L);
    // the transforms' first-pass reads stay in the stage, their exchanges in the group's buffer
    typedef KCSTile<L> Gm;
    for (int tid = 0; tid < Gm::NT; ++tid) {
        int j, g;
        for (int q = 0; q < SG::XI::Q0; ++q) {
            bmap<LAYOUT_COL, L, Gm::G, SG::XI::R0>(tid + q * Gm::NT, j, g);
            expect_true((j + (SG::XI::R0 - 1) * (L / SG::XI::R0)) * Gm::G + g < Gm::TE, "stage read", L);
        }
        for (int q = 0; q < SG::XF::Q0; ++q) {
            bmap<LAYOUT_COL, L, Gm::G, SG::XF::R0>(tid + q * Gm::NT, j, g);
            expect_true((j + (SG::XF::R0 - 1) * (L / SG::XF::R0)) * Gm::G + g < Gm::TE, "stage read", L);
        }
    }
}

// entries that tw_init writes and tw_get reads, against the room of the tile
template <class Gm, int L> void exact_table(size_t outer) {
    typedef Tw<float, L, Gm::EX> W;
    typedef TwDims<L> D;
    const size_t room = Gm::smem_bytes / sizeof(float2) - ((size_t)Gm::TE + (Gm::TE >> Gm::P::PSH) + 1) - outer;
    if (W::FULL) {
        expect_true(room == (size_t)L, "whole table", L);
    } else if (W::COMP) {
        expect_true(room == (size_t)D::NLO + 2 * D::NHI && D::NHI <= 32 && 32 % D::NHI == 0, "tables with residuals", L);
        for (int e = 0; e < L; ++e)
            expect_true((e >> D::SH) < D::NHI && tw_lo_slot<D::NLO>(e & (D::NLO - 1)) < D::NLO, "entries", L);
    } else {
        expect_true(room == (size_t)D::NLO + D::NHI, "two-level tables", L);
    }
}
template <int L> void tiles() {
    typedef KCGeom<float, L, 1> C1;
    typedef KCGeom<float, L, 2> C2;
    exact_table<C1, L>((size_t)C1::G * (C1::OLO + C1::OHI));
    exact_table<C2, L>((size_t)C2::G * (C2::OLO + C2::OHI));
    typedef KRGeom<float, L, 1> R1;
    typedef KRGeom<float, L, 2> R2;
    exact_table<R1, L>((size_t)R1::G * (R1::OLO + R1::OHI));
    exact_table<R2, L>((size_t)R2::G * (R2::OLO + R2::OHI));
    if constexpr (L >= 256) exact_table<KNGeom<float, L, 1>, L>(0);
}

static void w32_values() {
    for (int m = 0; m < 32; ++m) {
        const long double x = 2.0L * acosl(-1.0L) * m / 32;
        float2 hi, res;
        w32(m, hi, res);
        expect_true(std::fabs((double)(hi.x + (long double)res.x - cosl(x))) < 1e-14, "cos", m);
        expect_true(std::fabs((double)(hi.y + (long double)res.y - sinl(x))) < 1e-14, "sin", m);
        expect_true(std::fabs(res.x) <= 0x1p-25f && std::fabs(res.y) <= 0x1p-25f, "half a unit", m);
    }
}

// scatter of the first pass, reads and writes of pass P
template <int LAYOUT, int L, int G, int PSH, bool SF, int P> void slots() {
    typedef Sched<L, (1 << PSH)> SC;
    if constexpr (P < SC::NP) {
        typedef Slot<LAYOUT, L, G, PSH> SL;
        constexpr int R = SC::template radix<SF>(P), NS = SC::template ns<SF>(P);
        auto same = [](int lb, int c, int g) {
            expect_true(SL::base(lb, g) + SL::off(c) == phys<PSH>(eidx<LAYOUT, L, G>(lb + c, g)), "slot", L);
        };
        for (int j = 0; j < L / R; ++j)
            for (int g = 0; g < G; ++g)
                for (int r = 0; r < R; ++r) {
                    const int k = j & (NS - 1);
                    if (P == 0) same(j * R, r, g);
                    if (P > 0 && SL::template strided<L / R, R>()) same(j, r * (L / R), g);
                    if (P > 0 && P < SC::NP - 1 && SL::template strided<NS, R>()) same((j - k) * R + k, r * NS, g);
                }
        slots<LAYOUT, L, G, PSH, SF, P + 1>();
    }
}
template <int L> void fine64_slots() {
    typedef KCGeom<double, L, 1> C;
    typedef KRGeom<double, L, 1> R;
    static_assert(C::P::PSH == 2 && R::P::PSH == 2, "the fine FP64 tiles");
    slots<LAYOUT_COL, L, C::G, 2, true, 0>();
    slots<LAYOUT_COL, L, C::G, 2, false, 0>();
    slots<LAYOUT_ROW, L, R::G, 2, true, 0>();
    slots<LAYOUT_ROW, L, R::G, 2, false, 0>();
}

int main() {
    staged_direct_table<256>();
    staged_direct_table<512>();
    staged_direct_table<1024>();
    staged_direct_table<2048>();
    tiles<16>();
    tiles<32>();
    tiles<64>();
    tiles<128>();
    tiles<256>();
    tiles<512>();
    tiles<1024>();
    tiles<2048>();
    exact_table<KNGeom<float, 4096, 1>, 4096>(0);
    w32_values();
    fine64_slots<16>();
    fine64_slots<32>();
    fine64_slots<64>();
    fine64_slots<128>();
    fine64_slots<256>();
    fine64_slots<512>();
    fine64_slots<1024>();
    fine64_slots<2048>();
    std::printf("checked %lld\n", g_checked);
    return 0;
}
