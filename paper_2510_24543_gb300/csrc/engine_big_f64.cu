// Lengths 128 and 256 of Engine<double>.
#include "engine_ext.cuh"
EGPE_EXT_DEFINE(big, 128, 256)
EGPE_EXT_INSTANTIATE(double, big)
EGPE_EXT_INSTANTIATE_CARRIED(big)
