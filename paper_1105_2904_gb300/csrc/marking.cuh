// Per-entry steps of the incremental owner-map update, shared by the per-phase kernels of the
// particle phase (particles.cu) and the one-launch form for few particles (k_remark in
// sweep.cuh). Integer work only.
#pragma once

#include "kernels.h"

namespace lbmp {

// Clears the tag word of the float4 BS record of site (index site, coordinates v) when the site
// stops being a BS site of the particle that wrote it (the FP64 mode checks the owner map
// instead).
__device__ __forceinline__ void drop_record(const ParticleArgs& a, unsigned site, const int v[3])
{
    if (a.scratch_f64) return;
    const unsigned ri = a.rec_brick ? rec_brick_index(a.g, v[0], v[1], v[2]) : site;
    ((unsigned*)a.bs_scratch)[(size_t)ri * 4 + 3] = TAG_FLUID;
}

// Wrapped anchor of a particle before this step's move.
struct OldAnchor {
    int Kw[3];
    __device__ __forceinline__ OldAnchor(const ParticleArgs& a, int p)
    {
        const int K[3] = {a.Kold[(size_t)p * 3], a.Kold[(size_t)p * 3 + 1], a.Kold[(size_t)p * 3 + 2]};
        wrap_anchor(a.g, K, Kw);
    }
};

// Releases the site of template entry e if the moved particle p owned it at its old anchor.
__device__ __forceinline__ void clear_entry(const ParticleArgs& a, int p, const OldAnchor& o, int e)
{
    const int ent = a.tmpl[a.pc[p].tmpl_off + e];
    unsigned site;
    int v[3];
    if (!site_fast_xyz(a.g, o.Kw, tmpl_ox(ent), tmpl_oy(ent), tmpl_oz(ent), site, v)) return;
    const unsigned t = a.tag[site];
    if (t != TAG_FLUID && (t & PID_MASK) == (unsigned)p) {
        a.tag[site] = TAG_FLUID;
        if ((t >> 30) == CLS_BS) drop_record(a, site, v);
    }
}

// Claims the site of template entry e for particle p at its current anchor; the lowest code wins.
__device__ __forceinline__ void stamp_entry(const ParticleArgs& a, int p, int e)
{
    const int Kw[3] = {a.pk[p].Kw[0], a.pk[p].Kw[1], a.pk[p].Kw[2]};
    const int ent = a.tmpl[a.pc[p].tmpl_off + e];
    unsigned site;
    int v[3];
    if (!site_fast_xyz(a.g, Kw, tmpl_ox(ent), tmpl_oy(ent), tmpl_oz(ent), site, v)) return;
    const unsigned code = (tmpl_cls(ent) << 30) | (unsigned)p;
    const unsigned old = atomicMin(&a.tag[site], code);
    // a BS site taken over by a lower code is no longer its particle's BS site
    if (code < old && (old >> 30) == CLS_BS) drop_record(a, site, v);
}

}  // namespace lbmp
