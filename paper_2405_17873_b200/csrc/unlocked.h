// A call with Python's global interpreter lock released, which is held again afterwards, also when the call throws.
#pragma once

#include <Python.h>

template <typename F>
auto unlocked(F&& f)
{
    struct Released {
        PyThreadState* state = PyEval_SaveThread();
        ~Released() { PyEval_RestoreThread(state); }
    } released;
    return f();
}
