// What a test sees of the stand-ins in fake_cudart.cpp.
#pragma once
#include <string>
#include <vector>

void set_device(int dev);                // the calling thread's current device, 0 or 1
int multiprocessors(int dev);
std::vector<unsigned>& grids();          // grid sizes of the calling thread's launches
bool& tensor_maps();                     // whether the driver has cuTensorMapEncodeTiled
void finding(const std::string& what);   // prints and counts
int findings();
