// Host helpers shared between the single-lattice and the batch/serve parts of the C ABI.
#pragma once

#include <string>

#include "fmlbm.h"
#include "fmlbm_kernels.cuh"

// Appendix C constants of a mixture (a_i, b_i, alpha_i(T), (a alpha)_ij, kappa_ij);
// false with a reason when the mixture is invalid.
bool fmlbm_internal_mixture_constants(const fmlbm_mixture& m, fmlbm::MixConst* mc, std::string* why);
// Validity of a lattice description for n components.
bool fmlbm_internal_lattice_ok(const fmlbm_lattice& L, int nc, std::string* why);
// Device bytes of a lattice in a batch: fmlbm_lattice_bytes without a handle's own scratch.
size_t fmlbm_internal_batched_bytes(int nc, const fmlbm_lattice& L);
// A device (or managed) allocation on `device`, aligned to `align` bytes, with at least
// `bytes` from p to the end of the allocation that contains it.
bool fmlbm_internal_usable_device_pointer(const void* p, size_t bytes, int device, size_t align = 16);
// A slab of a decomposed lattice in the decomposition's buffers: without scratch of its own, and with
// the domain check of its steps restricted to rows [y0, y1), its own rows without the ghost rows.
fmlbm_status fmlbm_internal_create_slab(const fmlbm_mixture* mixture, const fmlbm_lattice* lattice, void* cuda_stream,
                                        void* const g[2], float* const g0[2], void* const force[2], int y0, int y1,
                                        fmlbm_handle** out);
// Bytes of the two-launch step's scratch planes for a lattice (0: it does not take that step), and
// planes for a handle that outlive it.  Handles that step one after the other on one stream may share them.
size_t fmlbm_internal_fields_bytes(int nc, const fmlbm_lattice& L);
void fmlbm_internal_lend_fields(fmlbm_handle* h, void* fields);
