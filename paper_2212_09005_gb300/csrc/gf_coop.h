// Cooperative launches where fewer CTAs fit than the device would hold. Host
// code without CUDA, so that the CPU tests can build it.
#pragma once

namespace gf {

// Launches `grid` CTAs whose kernel waits for all of them, whatever their number.
// A context or stream on a part of the SMs refuses a grid that is sized for the
// device: then with half as many, down to one. launch(grid) gives its error,
// forget() takes a refused launch's off the record. Returns the last launch's.
template <class Err, class Launch, class Forget>
Err coop_launch(int grid, Err refused, Launch launch, Forget forget)
{
    Err e = launch(grid);
    while (e == refused && grid > 1) {
        forget();
        grid /= 2;
        e = launch(grid);
    }
    return e;
}

}  // namespace gf
