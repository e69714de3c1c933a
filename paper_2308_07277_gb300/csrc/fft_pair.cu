// Host side of the FP32 FFT path on two transforms at once (kernels in fft_pair.cuh).
#include "fft_pair.cuh"

namespace qm {
using namespace pr;


bool pair_path(qm_gspace g, int ntr) {
    // pairs halve the CTAs: below two plane CTAs per SM the single transforms are faster
    if (ntr && (long)((ntr + 1) / 2) * g->n[0] < 2L * device_sms()) return false;
    for (int d = 0; d < 3; ++d)
        if (pair_class(g->n[d]) < 0) return false;
    return plane_smem(g) <= kPairSmem && stick_smem(g) <= kPairSmem;
}
size_t pair_unit_bytes(qm_gspace g, int ik) { return (size_t)g->n[0] * g->k[ik].nstick_pad * sizeof(c2); }

qm_status local_kinetic_pair(qm_gspace g, int ik, int nb, const void* psi, int ld_psi, const void* vt, void* out, int ld_out,
                             void* tbuf, size_t tbuf_bytes, cudaStream_t s, cudaEvent_t wait_k3, bool accumulate, bool gamma) {
    const KTables& kt = g->k[ik];
    const int N1 = g->n[0], N2 = g->n[1], N3 = g->n[2];
    if (gamma && !kt.gamma) return fail(QM_ERR_ARG, "FFT path: the k-point is not the Gamma point");
    const int per = gamma ? 4 : 2;  // bands per pair of transforms
    const int npair = (nb + per - 1) / per;
    const int chunk = (int)std::max<size_t>(1, std::min<size_t>({(size_t)npair, tbuf_bytes / pair_unit_bytes(g, ik), kMaxGridY}));
    const size_t sm_stick = stick_smem(g), sm_plane = plane_smem(g);
    const int bx = pair_class(N1), byz = std::max(pair_class(N2), pair_class(N3));
    auto kxi = bx ? k_pair_x_inverse<1> : k_pair_x_inverse<0>;
    auto kxf = bx ? k_pair_x_forward<1> : k_pair_x_forward<0>;
    auto kxg = bx ? k_pair_x_forward_gamma<1> : k_pair_x_forward_gamma<0>;
    auto kpl = byz ? k_pair_plane<1> : k_pair_plane<0>;
    qm_status st;
    if ((st = allow_dynamic_smem((const void*)kpl, sm_plane, "qm_hpsi: FFT planes in shared memory")) ||
        (st = allow_dynamic_smem((const void*)kxi, sm_stick, "qm_hpsi: FFT sticks in shared memory")) ||
        (st = allow_dynamic_smem(gamma ? (const void*)kxg : (const void*)kxf, sm_stick,
                                 "qm_hpsi: FFT sticks in shared memory")))
        return st;
    const int nt = plane_nt((const void*)kpl, sm_plane, byz);
    const int ntile = (kt.nstick + kPairTile - 1) / kPairTile;
    c2* T = (c2*)tbuf;
    for (int p0 = 0; p0 < npair; p0 += chunk) {
        const int np = std::min(chunk, npair - p0), b0 = per * p0, nbx = std::min(per * np, nb - b0);
        const float2* ps = (const float2*)psi + (size_t)b0 * ld_psi;
        float2* po = (float2*)out + (size_t)b0 * ld_out;
        {
            ProfScope pf(PF_STICK_INV, s);
            kxi<<<dim3(ntile, np), stick_nt(N1, false), sm_stick, s>>>(ps, ld_psi, nbx, gamma ? 1 : 0, kt.runs, kt.nstick,
                                                                           kt.nstick_pad, N1, g->tw32[0], g->ldx, T);
        }
        {
            ProfScope pf(PF_PLANE, s);
            kpl<<<dim3(N1, np), nt, sm_plane, s>>>(T, kt.nstick_pad, kt.ymap, kt.lo, kt.hi, N1, N2, N3, g->tw32[1],
                                                            g->tw32[2], g->ldy, (const float*)vt);
        }
        if (wait_k3 && p0 == 0) {
            cudaError_t e = cudaStreamWaitEvent(s, wait_k3, 0);
            if (e != cudaSuccess) return cuda_check(e, "FFT path: wait for the nonlocal part");
        }
        {
            ProfScope pf(PF_STICK_FWD, s);
            if (gamma)
                kxg<<<dim3(kt.ngtile, np), stick_nt(N1, true), sm_stick, s>>>(
                    T, nbx, kt.gtile, kt.stick_g0, kt.g_code, kt.nstick_pad, N1, g->tw32[0], g->ldx, kt.kin_f, ps, ld_psi, po,
                    ld_out, accumulate ? 1 : 0);
            else
                kxf<<<dim3(ntile, np), stick_nt(N1, true), sm_stick, s>>>(T, nbx, kt.runs, kt.nstick, kt.nstick_pad, N1,
                                                                               g->tw32[0], g->ldx, kt.kin_f, ps, ld_psi, po, ld_out,
                                                                               accumulate ? 1 : 0);
        }
    }
    return cuda_check(cudaGetLastError(), "FFT path launch");
}

}  // namespace qm
