// Device view of a host-side operator.
#pragma once
#include "bttb_kernels.cuh"
#include "gj_internal.h"

namespace gj {

template <typename R>
inline OpView<R> view_of(const gj_op *op) {
    OpView<R> v;
    v.sx = op->sx; v.sy = op->sy; v.nx = op->nx; v.ny = op->ny; v.nz = op->nz;
    v.Nx = op->Nx; v.Ny = op->Ny; v.ncol = op->ncol;
    v.px = op->px; v.py = op->py;
    v.twx = static_cast<const cpx<R> *>(op->twx);
    v.twy = static_cast<const cpx<R> *>(op->twy);
    v.spec = static_cast<const cpx<R> *>(op->spec);
    v.Z = static_cast<cpx<R> *>(op->Z);
    // the recompute mode keeps no spectra: the plane they would take holds the layer sum
    v.Y = static_cast<cpx<R> *>(op->recompute ? op->spec : op->Y);
    v.W = static_cast<cpx<R> *>(op->W);
    v.V = static_cast<cpx<R> *>(op->V);
    v.cnt = op->cnt;
    v.real_spec = op->real_spec ? 1 : 0;
    v.tcol = op->fast1024 ? op->Ny / 2 : 0;
    v.split_half = op->fast || op->fast1024;  // the general kernels' spectra carry the factor
    return v;
}

// Shared memory of a row pass (two buffers of P lines and the twiddles) and of a column
// pass (two buffers of B lines, `keep` more lines that stay, the twiddles).
inline size_t row_smem(int Nx, int pitch, size_t cs) { return (size_t)(2 * Nx * pitch + Nx) * cs; }
inline size_t col_smem(int Ny, int pitch, int keep, size_t cs) { return (size_t)(2 * Ny * pitch + Ny * keep + Ny) * cs; }

}  // namespace gj
