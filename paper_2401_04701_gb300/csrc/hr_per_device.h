// hr_per_device.h - launch state that belongs to a device.
#pragma once

#include <mutex>

// One T for each CUDA device of the process, made on the first call for that device.
// Occupancy, SM counts and kernel attributes (a kernel with more than 48 KB of dynamic
// shared memory does not launch without its attribute) hold for the device they were
// asked for or set on; threads may come at once.
template <class T>
class hr_per_device {
    static constexpr int MAX = 64;
    std::once_flag once[MAX];
    T value[MAX];

public:
    template <class F>
    T get(int device, F make)
    {
        if (device < 0 || device >= MAX) return make();
        std::call_once(once[device], [&] { value[device] = make(); });
        return value[device];
    }
};
