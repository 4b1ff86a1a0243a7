// ffno_place.h -- which caller buffers the factorised surrogate's kernels read
// and write where they are (host code).
#pragma once
#include <cuda_runtime_api.h>

namespace ffno {

enum Place {
    PLACE_HOST,          // copied; results are waited for
    PLACE_ELSEWHERE,     // memory of another device: copied on the stream (its pages need not be mapped here)
    PLACE_HERE           // used in place
};

inline Place place_of(const cudaPointerAttributes &at, int device)
{
    if (at.type == cudaMemoryTypeManaged) return PLACE_HERE;
    if (at.type != cudaMemoryTypeDevice) return PLACE_HOST;
    return at.device == device ? PLACE_HERE : PLACE_ELSEWHERE;
}

}  // namespace ffno
