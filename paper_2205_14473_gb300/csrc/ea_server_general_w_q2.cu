// The staged server of messages with short blocks or with groups that span tiles: Adam at the workers, broadcast kind QK_UNIF.
#include "ea_server_general.cuh"
namespace ea {
template cudaError_t launch_server_general<MODE_W, QK_UNIF>(const ServerArgs &a, cudaStream_t s);
}
