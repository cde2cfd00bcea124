// The staged server of messages with short blocks or with groups that span tiles: Adam at the server, broadcast kind QK_POW2.
#include "ea_server_general.cuh"
namespace ea {
template cudaError_t launch_server_general<MODE_S, QK_POW2>(const ServerArgs &a, cudaStream_t s);
}
