// Mixed-radix lengths 48 and 96 of Engine<double>.
#include "engine_ext.cuh"
EGPE_EXT_DEFINE(mr, 48, 96)
EGPE_EXT_INSTANTIATE(double, mr)
EGPE_EXT_INSTANTIATE_CARRIED(mr)
