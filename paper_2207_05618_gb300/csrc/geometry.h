// Device geometry of a mesh, shared by the rendering and displacement
// kernels (raster.cu, displace.cu).
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

// The intrinsic triangle of each halfedge (paper Alg. 1) is evaluated once,
// when the geometry is made: 48 bytes per halfedge, three 16-byte words
//   (v0.x, v0.y, v0.z, Vert(Next h)), (v1.x, v1.y, v1.z, Face(h)),
//   (v2.x, v2.y, v2.z, Vert(h))
// (the ids as int bits), so that no kernel walks the face cycle per pixel or
// per lattice point.
struct htex_geometry {
    int32_t H = 0, V = 0, F = 0;
    float4* d_tri = nullptr;     // [H][3]
    float* d_vn = nullptr;       // [V][3] vertex normals
    float* d_fn = nullptr;       // [F][3] face normals
};
