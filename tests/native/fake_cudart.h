// fake_cudart.h -- what a test sees of the stand-in runtime.
#pragma once

extern thread_local int fake_device;        // the current device
extern int fake_placeable[4];               // largest cluster of each device
extern int fake_launches, fake_refused;     // launches taken and refused
extern int fake_cluster;                    // blocks of the last cluster launch
