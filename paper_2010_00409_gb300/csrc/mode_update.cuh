// The per-mode update of the generic k-space passes (kspace.cu, fft_two.cuh), every
// KspaceMode: Eq. 3-4 of Sec. 2.1, or the transverse projection alone.
#pragma once

#include "common.cuh"

namespace psatd {

template <typename T>
__device__ __forceinline__ void mode_update(cplx<T>* F0, cplx<T>* F1, cplx<T>* F2, cplx<T>* F3,
                                            cplx<T>* F4, cplx<T>* F5, T nx, T ny, T nz, T C, T S,
                                            int mode, T scale) {
    const cplx<T> Ex = *F0, Ey = *F1, Ez = *F2;
    cplx<T> Bx = *F3, By = *F4, Bz = *F5;
    if (mode == KS_ROTATE_SPECTRAL_PROJ) {
        const cplx<T> kB = mk<T>(nx * Bx.x + ny * By.x + nz * Bz.x, nx * Bx.y + ny * By.y + nz * Bz.y);
        Bx = csub(Bx, cscale(kB, nx));
        By = csub(By, cscale(kB, ny));
        Bz = csub(Bz, cscale(kB, nz));
    }
    if (mode == KS_PROJECT) {
        cplx<T> kE = mk<T>(nx * Ex.x + ny * Ey.x + nz * Ez.x, nx * Ex.y + ny * Ey.y + nz * Ez.y);
        cplx<T> kB = mk<T>(nx * Bx.x + ny * By.x + nz * Bz.x, nx * Bx.y + ny * By.y + nz * Bz.y);
        *F0 = cscale(csub(Ex, cscale(kE, nx)), scale);
        *F1 = cscale(csub(Ey, cscale(kE, ny)), scale);
        *F2 = cscale(csub(Ez, cscale(kE, nz)), scale);
        *F3 = cscale(csub(Bx, cscale(kB, nx)), scale);
        *F4 = cscale(csub(By, cscale(kB, ny)), scale);
        *F5 = cscale(csub(Bz, cscale(kB, nz)), scale);
        return;
    }
    const cplx<T> kE = mk<T>(nx * Ex.x + ny * Ey.x + nz * Ez.x, nx * Ex.y + ny * Ey.y + nz * Ez.y);
    // n x B and n x E
    const cplx<T> cBx = mk<T>(ny * Bz.x - nz * By.x, ny * Bz.y - nz * By.y);
    const cplx<T> cBy = mk<T>(nz * Bx.x - nx * Bz.x, nz * Bx.y - nx * Bz.y);
    const cplx<T> cBz = mk<T>(nx * By.x - ny * Bx.x, nx * By.y - ny * Bx.y);
    const cplx<T> cEx = mk<T>(ny * Ez.x - nz * Ey.x, ny * Ez.y - nz * Ey.y);
    const cplx<T> cEy = mk<T>(nz * Ex.x - nx * Ez.x, nz * Ex.y - nx * Ez.y);
    const cplx<T> cEz = mk<T>(nx * Ey.x - ny * Ex.x, nx * Ey.y - ny * Ex.y);
    // i S v = (-S v.y, S v.x)
    *F0 = mk<T>(C * (Ex.x - nx * kE.x) - S * cBx.y, C * (Ex.y - nx * kE.y) + S * cBx.x);
    *F1 = mk<T>(C * (Ey.x - ny * kE.x) - S * cBy.y, C * (Ey.y - ny * kE.y) + S * cBy.x);
    *F2 = mk<T>(C * (Ez.x - nz * kE.x) - S * cBz.y, C * (Ez.y - nz * kE.y) + S * cBz.x);
    *F3 = mk<T>(C * Bx.x + S * cEx.y, C * Bx.y - S * cEx.x);
    *F4 = mk<T>(C * By.x + S * cEy.y, C * By.y - S * cEy.x);
    *F5 = mk<T>(C * Bz.x + S * cEz.y, C * Bz.y - S * cEz.x);
}

}  // namespace psatd
