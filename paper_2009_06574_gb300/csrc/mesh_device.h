// The mesh tables of mesh_host.h, found on the device (k_mesh.cu).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace hexfc {

// The device memory of one mesh's tables while they are found. Both calls work on
// the legacy default stream and wait for it; *host: the tables are to be found on
// the host instead (a vertex of extreme valence, or cells that list a face's
// corners in different orders).
struct MeshScratch {
    void* block = nullptr;
    uint64_t *scal = nullptr, *foff = nullptr, *eoff = nullptr;
    uint4* fsort = nullptr;
    uint2* esort = nullptr;
    uint32_t *fnum = nullptr, *enum_ = nullptr;

    MeshScratch() = default;
    MeshScratch(const MeshScratch&) = delete;
    MeshScratch& operator=(const MeshScratch&) = delete;
    ~MeshScratch();
    // Sorts and numbers the faces and edges of the (valid) cells.
    cudaError_t number(const int32_t* cells, int64_t n_cells, int64_t n_verts, uint64_t* n_faces, uint64_t* n_edges, bool* host);
    // Writes the tables; level: [12 C] of the cells' edges, nullptr: all 0.
    cudaError_t write(const int32_t* cells, int64_t n_cells, const uint8_t* level, int32_t* cell_edges, uint8_t* elevel,
                      int4* fverts, int4* fedges, uint8_t* fbound, bool* host);
};

}  // namespace hexfc
