// The device buffers that the host-buffer entry point keeps with an operator
// (hho_erk_run_host): its state and canonical vector, and a work buffer that
// grows with the tableau.  Apart from the CUDA calls, so that a failed allocation
// can be tried on the host.
#pragma once

#include "hho_internal.h"

// Makes the buffers that are missing or too small.  alloc(size_t doubles) returns
// nullptr on failure, release(double*) frees, zero(double*, size_t doubles) says
// whether it could queue the clearing.  After a failure what is kept is
// consistent: every pointer is null or a whole buffer, host_work_size is that of
// the buffer in d_host_work, and the next call takes up what is missing.  *made:
// a buffer is new.
template <class Alloc, class Release, class Zero>
int grow_host_buffers(hho_ops* ops, int64_t work_size, Alloc alloc, Release release, Zero zero, bool* made) {
    *made = !ops->d_host_state || !ops->d_host_canon || ops->host_work_size < work_size;
    if (!ops->d_host_state && !(ops->d_host_state = alloc((size_t)ops->n_state))) return HHO_ENOMEM;
    if (!ops->d_host_canon && !(ops->d_host_canon = alloc((size_t)ops->n_canonical))) return HHO_ENOMEM;
    if (ops->host_work_size >= work_size) return HHO_OK;
    if (ops->d_host_work) release(ops->d_host_work);
    ops->host_work_size = 0;
    if (!(ops->d_host_work = alloc((size_t)work_size))) return HHO_ENOMEM;
    // the mapped path leaves padding slots of its states unwritten
    if (!zero(ops->d_host_work, (size_t)work_size) || !zero(ops->d_host_state, (size_t)ops->n_state)) return HHO_ECUDA;
    ops->host_work_size = work_size;
    return HHO_OK;
}
