// Makes the launch plans of every batch size on the host (no device: the tensor maps are not encoded) and checks what holds for all of
// them.  Prints one line per violation; exit code 1 if there is one.
#include "../paper_1412_2302_b200/csrc/alexnet_api.cu"

static CUresult CUDAAPI no_encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
    return CUDA_SUCCESS;
}
static int columns(int n) { int c = 32; while (c < n) c <<= 1; return c; }      // as the kernels allocate them

int main() {
    const uint32_t forms[3] = {0, ALEXNET_FLAG_NO_CTA_PAIRS, ALEXNET_FLAG_ALL_CTA_PAIRS};
    int bad = 0;
    for (uint32_t flags : forms)
        for (int B = 1; B <= 1024; ++B) {
            alexnet h{};
            h.cfg.batch = B; h.cfg.replicas = 1; h.cfg.lrn_size = 5; h.cfg.lrn_k = 2.f; h.cfg.flags = flags;
            h.B = B; h.L = make_layout(); h.sm_count = kSms; h.encode = no_encode;
            carve(&h, (uint8_t*)1024);
            if (build_plans(&h, 0)) { printf("batch %d flags %u: no plan\n", B, flags); return 1; }
            const Replica& R = h.rep[0];
            auto check = [&](const char* name, int l, const Plan& P) {
                const int cols = P.conv ? columns(P.c.acc_stages * P.c.MH * P.c.BN)
                                 : P.wgrad ? columns((P.w.solo ? 2 : 1) * 64 * (P.w.kw_parts == 2 ? std::max(P.w.acc_taps[0], P.w.acc_taps[1]) : P.w.kw))
                                 : P.upd ? 2 * tc::kUpdBN : columns(2 * P.p.BN);
                // two CTAs (and the 1 KB of each that the system takes) do not fit in the 228 KB of an SM, one does
                const bool alone = 2 * (P.smem + 1024) > 228 * 1024, fits = P.smem <= 227 * 1024;
                if (!alone || !fits || cols > 512) {
                    printf("batch %d flags %u %s %d: %zu bytes of shared memory, %d columns\n", B, flags, name, l + 1, P.smem, cols);
                    bad = 1;
                }
            };
            for (int l = 0; l < 5; ++l) {
                check("conv forward", l, R.conv_fwd[l][0]); check("conv backward-data", l, R.conv_bwd[l]);
                check("conv backward-data beside the updates", l, R.conv_bwd_beside[l]); check("conv weight gradient", l, R.conv_wg[l][0]);
            }
            for (int l = 0; l < 3; ++l) {
                check("FC forward", l, R.fc_fwd[l]); check("FC backward-data", l, R.fc_bwd[l]);
                check("FC weight gradient", l, R.fc_wg_plain[l]); check("FC update", l, R.fc_upd[l]);
            }
        }
    if (2 * (tc::fc_chain_smem_bytes() + 1024) <= 228 * 1024) { printf("FC chain\n"); bad = 1; }
    return bad;
}
