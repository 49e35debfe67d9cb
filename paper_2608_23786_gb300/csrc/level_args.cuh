// A context as the level arguments of the stepper kernels.
#pragma once
#include "internal.h"
#include "stepper_impl.cuh"

namespace mclbm {

inline Geom geom_of(const mclbm_ctx* c) { return Geom{c->N, c->logN, c->n}; }
inline int parity_of(const mclbm_ctx* c) { return c->cfg.pattern == MCLBM_AA ? (int)(c->steps & 1) : 0; }

template <class E>
void fill_level(LevelArgs<E>& L, const mclbm_ctx* c)
{
    if (c->cfg.pattern == MCLBM_PULL) {
        L.src = (const E*)lattice_ptr(c, c->cur);
        L.dst = (E*)lattice_ptr(c, 1 - c->cur);
    } else {
        L.src = (const E*)lattice_ptr(c, 0);
        L.dst = (E*)lattice_ptr(c, 0);
    }
    L.g = geom_of(c);
    L.M = c->M;
    L.parity = parity_of(c);
    L.omega32 = (float)c->units.omega;
    L.omega64 = c->units.omega;
    L.a32 = (float)(2.0 / c->units.omega);
    L.b32 = (float)(2.0 - 2.0 / c->units.omega);
    if constexpr (std::is_same<E, double>::value) {
        L.a64 = 2.0 / c->units.omega;
        L.b64 = 2.0 - 2.0 / c->units.omega;
    }
}

}  // namespace mclbm
