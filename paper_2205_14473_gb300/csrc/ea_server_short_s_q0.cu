// The staged server of messages with several scales per tile: Adam at the server, broadcast kind QK_IDENT.
#include "ea_server_short.cuh"
namespace ea {
template cudaError_t launch_server_short<MODE_S, QK_IDENT>(const ServerArgs &a, cudaStream_t s);
}
