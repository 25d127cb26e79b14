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

// A listed particle as the re-marking kernels use it, loaded once for all of its entries: its template
// entries (BS, IS, interior from off on, n in all) and its wrapped anchor.
struct Stamped {
    int p, off, n;
    int Kw[3];
    Stamped() = default;
    __device__ __forceinline__ Stamped(const PConst* pc, const PKern* pk, int q)
        : p(q), off(pc[q].tmpl_off), n(pc[q].tmpl_n), Kw{pk[q].Kw[0], pk[q].Kw[1], pk[q].Kw[2]}
    {
    }
};

// The same for a particle whose shift changed, with its IS entries (n_is from is_off on) and the
// wrapped anchor before the move.
struct Moved : Stamped {
    int is_off, n_is;
    int Ko[3];
    Moved() = default;
    __device__ __forceinline__ Moved(const Geom& g, const PConst* pc, const PKern* pk, const int* Kold, int q)
        : Stamped(pc, pk, q), is_off(pc[q].tmpl_off + pc[q].n_bs), n_is(pc[q].n_is)
    {
        const int K[3] = {Kold[(size_t)q * 3], Kold[(size_t)q * 3 + 1], Kold[(size_t)q * 3 + 2]};
        wrap_anchor(g, K, Ko);
    }
};

// Template entries e, e + step, ... of a particle (U of them, those below h.n; the others fluid) and
// their sites at the wrapped anchor K; ok: inside the domain. The U loads are in flight together.
template <int U>
struct EntrySites {
    int ent[U], v[U][3];
    unsigned site[U];
    bool ok[U];
    __device__ __forceinline__ EntrySites(const Geom& g, const int* tmpl, const Stamped& h, const int K[3], int e, int step)
    {
#pragma unroll
        for (int u = 0; u < U; ++u) ent[u] = e + u * step < h.n ? tmpl[h.off + e + u * step] : 0;
#pragma unroll
        for (int u = 0; u < U; ++u)
            ok[u] = site_fast_xyz(g, K, tmpl_ox(ent[u]), tmpl_oy(ent[u]), tmpl_oz(ent[u]), site[u], v[u]) && e + u * step < h.n;
    }
};

// Releases the sites of entries e, e + step, ... that the moved particle owned at its old anchor.
template <int U>
__device__ __forceinline__ void clear_entries(const ParticleArgs& a, const Moved& h, int e, int step)
{
    const EntrySites<U> s(a.g, a.tmpl, h, h.Ko, e, step);
    unsigned t[U];
#pragma unroll
    for (int u = 0; u < U; ++u) t[u] = s.ok[u] ? a.tag[s.site[u]] : TAG_FLUID;
#pragma unroll
    for (int u = 0; u < U; ++u)
        if (t[u] != TAG_FLUID && (t[u] & PID_MASK) == (unsigned)h.p) {
            a.tag[s.site[u]] = TAG_FLUID;
            if ((t[u] >> 30) == CLS_BS) drop_record(a, s.site[u], s.v[u]);
        }
}

// Claims the sites of entries e, e + step, ... for the particle at its current anchor; the lowest code
// wins.
template <int U>
__device__ __forceinline__ void stamp_entries(const ParticleArgs& a, const Stamped& h, int e, int step)
{
    const EntrySites<U> s(a.g, a.tmpl, h, h.Kw, e, step);
    unsigned code[U], old[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        code[u] = (tmpl_cls(s.ent[u]) << 30) | (unsigned)h.p;
        old[u] = s.ok[u] ? atomicMin(&a.tag[s.site[u]], code[u]) : code[u];
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
        // a BS site taken over by a lower code is no longer its particle's BS site
        if (code[u] < old[u] && (old[u] >> 30) == CLS_BS) drop_record(a, s.site[u], s.v[u]);
}

}  // namespace lbmp
