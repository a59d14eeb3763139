// Receiver geometry shared by the edge kernels.
#pragma once
#include "mp.cuh"

namespace dmts {

struct AtomGeom {
    float x, y, z, bx, by, bz, ibx, iby, ibz;
};

// The wi-th atom in processing order: index, row bounds, position and box.
struct Row {
    int i, beg, end;
    AtomGeom a;
};

__device__ __forceinline__ Row load_row(const EdgeGeom &g, int wi) {
    Row r;
    r.i = r.beg = r.end = 0;
    if (wi >= g.n_atoms) return r;
    const int i = g.order ? __ldg(g.order + wi) : wi;
    const int rep = g.atom_rep[i];
    r.i = i;
    r.beg = g.row_ptr[i];
    r.end = g.row_ptr[i + 1];
    r.a.x = g.x[3 * i]; r.a.y = g.x[3 * i + 1]; r.a.z = g.x[3 * i + 2];
    r.a.bx = g.box[3 * rep]; r.a.by = g.box[3 * rep + 1]; r.a.bz = g.box[3 * rep + 2];
    return r;
}

__device__ __forceinline__ AtomGeom wrap_inverse(AtomGeom a) {
    // an approximate reciprocal: it only picks the image, and the images are
    // equally far apart (half a box, beyond any cutoff) where that could differ
    a.ibx = a.bx > 0.f ? __fdividef(1.f, a.bx) : 0.f;
    a.iby = a.by > 0.f ? __fdividef(1.f, a.by) : 0.f;
    a.ibz = a.bz > 0.f ? __fdividef(1.f, a.bz) : 0.f;
    return a;
}

// Displacement x_j - x_i (minimum image) and its square, rounded the same way
// in every kernel that uses them and exactly antisymmetric / symmetric in
// (i, j): kernels that must agree on which edges are active use these.
__device__ __forceinline__ float4 edge_disp(const AtomGeom &a, float x, float y, float z) {
    float4 d = make_float4(x - a.x, y - a.y, z - a.z, 0.f);
    d.x = fmaf(-a.bx, rintf(__fmul_rn(d.x, a.ibx)), d.x);   // an open axis has bx = ibx = 0
    d.y = fmaf(-a.by, rintf(__fmul_rn(d.y, a.iby)), d.y);
    d.z = fmaf(-a.bz, rintf(__fmul_rn(d.z, a.ibz)), d.z);
    d.w = fmaf(d.x, d.x, fmaf(d.y, d.y, __fmul_rn(d.z, d.z)));
    return d;
}

}  // namespace dmts
