"""No C++ exception leaves an entry point of the C ABI, and none that passes the binding's library call leaves Python's
global interpreter lock released."""
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2405_17873_b200", "csrc")


def _python(code, *args):
    return subprocess.run([sys.executable, "-c", code, *args], cwd=os.path.dirname(HERE), capture_output=True, text=True,
                          env=dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(HERE), HERE])))


def test_layer_call_without_memory_for_the_library_s_own_notes(recorded_library):
    run = _python("""
import sys
from recorded import BUFFER, Recorded
lib = Recorded(sys.argv[1])
layer = lambda: lib.so.mixdq_linear_q8(BUFFER, 64, 128, BUFFER, 64, 8, BUFFER, BUFFER, None, BUFFER, None, None)
lib.so.fake_fail_alloc(1)
rc = layer()
lib.so.fake_fail_alloc(0)
print(rc, lib.so.fake_launches(), layer())
""", recorded_library)
    assert run.returncode == 0 and run.stdout.split() == ["0", "1", "0"], (run.returncode, run.stdout, run.stderr)


def test_lock_is_held_again_behind_a_call_that_throws(tmp_path):
    source = tmp_path / "throws.cpp"
    source.write_text("""
#include <new>
#include "unlocked.h"
static PyObject* run(PyObject*, PyObject*)
{
    int inside = -1;
    try {
        unlocked([&]() -> int { inside = PyGILState_Check(); throw std::bad_alloc(); });
    } catch (const std::bad_alloc&) {
    }
    return Py_BuildValue("ii", inside, PyGILState_Check());
}
static PyMethodDef methods[] = {{"run", run, METH_NOARGS, nullptr}, {}};
static PyModuleDef module = {PyModuleDef_HEAD_INIT, "throws", nullptr, -1, methods};
PyMODINIT_FUNC PyInit_throws() { return PyModule_Create(&module); }
""")
    subprocess.run(["g++", "-std=c++17", "-fPIC", "-shared", "-I" + CSRC, "-I" + sysconfig.get_paths()["include"], str(source),
                    "-o", str(tmp_path / "throws.so")], check=True)
    run = _python("import sys; sys.path.insert(0, sys.argv[1]); import throws; print(*throws.run())", str(tmp_path))
    assert run.stdout.split() == ["0", "1"], (run.returncode, run.stdout, run.stderr)
