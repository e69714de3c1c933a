// GW matrix elements on the paired FP32 FFT path (kernels in fft_pair.cuh): host side.
#include "fft_pair.cuh"

namespace qm {
using namespace pr;

qm_status gw_mel_pair(qm_gspace g, int ikl, int ikr, int nl, const void* psi_l, int ld_l, int nr, const void* psi_r, int ld_r,
                      qm_gspace ge, int iq, void* M, int ld_m, cudaStream_t s) {
    const int N1 = g->n[0], N2 = g->n[1], N3 = g->n[2];
    const size_t nrr = (size_t)N1 * N2 * N3;
    const KTables &kl = g->k[ikl], &kr = g->k[ikr], &ke = ge->k[iq];
    const size_t sm_stick = stick_smem(g), sm_plane = plane_smem(g);
    const int bx = pair_class(N1), byz = std::max(pair_class(N2), pair_class(N3));
    auto kxi = bx ? k_pair_x_inverse<1> : k_pair_x_inverse<0>;
    auto kme = bx ? k_pair_mel<1> : k_pair_mel<0>;
    auto kre = byz ? k_pair_real<1> : k_pair_real<0>;
    auto kpr = byz ? k_pair_product<1> : k_pair_product<0>;
    qm_status st;
    if ((st = allow_dynamic_smem((const void*)kxi, sm_stick, "qm_gw_mel: sticks in shared memory")) ||
        (st = allow_dynamic_smem((const void*)kme, sm_stick, "qm_gw_mel: sticks in shared memory")) ||
        (st = allow_dynamic_smem((const void*)kre, sm_plane, "qm_gw_mel: planes in shared memory")) ||
        (st = allow_dynamic_smem((const void*)kpr, sm_plane, "qm_gw_mel: planes in shared memory")))
        return st;
    const int nt_re = plane_nt((const void*)kre, sm_plane, byz), nt_pr = plane_nt((const void*)kpr, sm_plane, byz);
    // workspace: left boxes (single) | right boxes (packed pairs) | stick buffer of the states | of the jobs
    constexpr size_t kChunk = 256ull << 20;
    const int nlp = (nl + 1) / 2, nrp = (nr + 1) / 2, njob = nl * nrp;
    const size_t per_t = (size_t)N1 * std::max(kl.nstick_pad, kr.nstick_pad) * sizeof(c2);
    const size_t per_e = (size_t)N1 * ke.nstick_pad * sizeof(c2);
    const int nbc = (int)std::max<size_t>(1, std::min<size_t>({(size_t)std::max(nlp, nrp), kChunk / per_t, kMaxGridY}));
    const int njc = (int)std::max<size_t>(1, std::min<size_t>({(size_t)njob, kChunk / per_e, kMaxGridY}));
    const size_t off_ul = kWsHeader;
    const size_t off_ur = align_up(off_ul + (size_t)nl * nrr * sizeof(float2), 256);
    const size_t off_t = align_up(off_ur + (size_t)nrp * nrr * sizeof(c2), 256);
    const size_t off_e = align_up(off_t + (size_t)nbc * per_t, 256);
    if ((st = ensure_workspace(g, align_up(off_e + (size_t)njc * per_e, 256), s))) return st;
    char* ws = (char*)g->ws.ptr;
    float2* UL = (float2*)(ws + off_ul);
    c2 *UR = (c2*)(ws + off_ur), *T = (c2*)(ws + off_t), *Te = (c2*)(ws + off_e);
    for (int side = 0; side < 2; ++side) {
        const KTables& kt = side ? kr : kl;
        const float2* psi = (const float2*)(side ? psi_r : psi_l);
        const int ld = side ? ld_r : ld_l, n = side ? nr : nl, np = side ? nrp : nlp;
        for (int p0 = 0; p0 < np; p0 += nbc) {
            const int npx = std::min(nbc, np - p0), nbx = std::min(2 * npx, n - 2 * p0);
            {
                ProfScope pf(PF_STICK_INV, s);
                kxi<<<dim3((kt.nstick + kPairTile - 1) / kPairTile, npx), stick_nt(N1, false), sm_stick, s>>>(
                    psi + (size_t)(2 * p0) * ld, ld, nbx, 0, kt.runs, kt.nstick, kt.nstick_pad, N1, g->tw32[0], g->ldx, T);
            }
            {
                ProfScope pf(PF_PLANE, s);
                kre<<<dim3(N1, npx), nt_re, sm_plane, s>>>(T, kt.nstick_pad, kt.ymap, kt.lo, kt.hi, N1, N2, N3, g->tw32[1],
                                                                   g->tw32[2], g->ldy, side ? UR + (size_t)p0 * nrr : nullptr,
                                                                   side ? nullptr : UL + (size_t)(2 * p0) * nrr, nbx);
            }
        }
    }
    const int ntile = (ke.nstick + kPairTile - 1) / kPairTile;
    for (int j0 = 0; j0 < njob; j0 += njc) {
        const int nj = std::min(njc, njob - j0);
        {
            ProfScope pf(PF_PLANE, s);
            kpr<<<dim3(nj, N1), nt_pr, sm_plane, s>>>(UL, UR, nrp, j0, Te, ke.nstick_pad, ke.ymap, ke.lo, ke.hi, N1, N2, N3,
                                                                 g->tw32[1], g->tw32[2], g->ldy);
        }
        {
            ProfScope pf(PF_STICK_FWD, s);
            kme<<<dim3(ntile, nj), stick_nt(N1, true), sm_stick, s>>>(Te, nr, nrp, j0, ke.runs, ke.nstick, ke.nstick_pad, N1,
                                                                     g->tw32[0], g->ldx, (float)(1.0 / (double)nrr), (float2*)M, ld_m);
        }
    }
    return cuda_check(cudaGetLastError(), "qm_gw_mel launch");
}

}  // namespace qm
