// ls_fft_widedf.cu -- the LS-apply and the incident right-hand side (Sec. 2) in double-float
// arithmetic, P >= 64 (ls_fft_wide.cuh).
#include "ls_fft_wide.cuh"

int ls_widedf_init() {
    LS_TRY((wide_optin<cdp, cdfl, SrcMU<dfl, double2>, DstApply<double2>>()));
    return wide_optin<cdp, cdfl, SrcIncDf, DstRhs>();
}
int ls_widedf_apply(ls_handle* h, const double2* u, double2* y) {
    return wide_apply<cdp>(h, SrcMU<dfl, double2>{h->mdf, u, h->n}, DstApply<double2>{u, y, h->n}, h->ghatdf, h->twwdf);
}
int ls_widedf_rhs(ls_handle* h, double2* f) {
    return wide_apply<cdp>(h, SrcIncDf{h->mdf, h->incxdf, h->inczdf, h->n}, DstRhs{f, h->n}, h->ghatdf, h->twwdf);
}
