// ls_fft_wide64.cu -- the LS-apply and the incident right-hand side (Sec. 2) in FP64, P >= 64
// (ls_fft_wide.cuh).
#include "ls_fft_wide.cuh"

int ls_wide64_init() {
    LS_TRY((wide_optin<double2, double2, SrcMU<double, double2>, DstApply<double2>>()));
    return wide_optin<double2, double2, SrcInc<double>, DstRhs>();
}
int ls_wide64_apply(ls_handle* h, const double2* u, double2* y) {
    return wide_apply<double2>(h, SrcMU<double, double2>{h->m64, u, h->n}, DstApply<double2>{u, y, h->n}, h->ghat64, h->tww64);
}
int ls_wide64_rhs(ls_handle* h, double2* f) {
    return wide_apply<double2>(h, SrcInc<double>{h->m64, h->incx, h->incz, h->n}, DstRhs{f, h->n}, h->ghat64, h->tww64);
}
