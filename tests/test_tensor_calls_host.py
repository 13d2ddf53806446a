"""What PagedAttention's calls with tensors refuse before they reach the device, against the calls through addresses."""
import os
import subprocess
import sys
import sysconfig

import numpy as np
import pytest
import torch

import paper_2507_17769_b200 as ps
from paper_2507_17769_b200 import session


def host_session():
    """A PagedAttention without a pool: what its calls do up to the library, which refuses a null pool before any device call."""
    pa = object.__new__(ps.PagedAttention)
    pa.torch, pa._calls = torch, ps.binding.calls()
    pa._tensor_calls, pa._tensor = session.torch_calls(), torch.Tensor
    pa.device, pa.shape = torch.device("cpu"), ps.binding.make_shape(8, 2, 64)
    pa.pool, pa.kv, pa._plan = torch.empty(16, dtype=torch.uint8), 0, None
    pa._stream = lambda: 0
    return pa


class Sub(torch.Tensor):  # (these take the calls through addresses)
    pass


@pytest.mark.parametrize("length", [2.5, np.float64(2), True, "3", None, torch.tensor(2.5)], ids=repr)
def test_gather_takes_no_length_that_is_not_an_integer(length):
    row = torch.zeros(4, dtype=torch.int32)
    for table in (row, row.as_subclass(Sub)):
        with pytest.raises(TypeError):
            host_session().gather(table, length)


def test_lengths_of_integer_types_are_taken():
    row = torch.zeros(4, dtype=torch.int32)
    for length in (3, np.int64(3), np.int32(3), torch.tensor(3)):
        for table in (row, row.as_subclass(Sub)):
            with pytest.raises(ps.PsError) as e:  # (as far as the null pool)
                host_session().gather(table, length)
            assert e.value.status == ps.binding.PS_ERR_INVALID


def test_a_closed_pool_is_reported_as_the_library_does():
    pa = host_session()
    pa.kv = None
    k, row = torch.zeros((1, 2, 64), dtype=torch.bfloat16), torch.zeros((1, 4), dtype=torch.int32)
    for cast in (lambda x: x, lambda x: x.as_subclass(Sub)):
        for call in (lambda: pa.write(cast(k), cast(k), cast(row), [0], [1]), lambda: pa.gather(cast(row), 1)):
            with pytest.raises(ps.PsError) as e:
                call()
            assert e.value.status == ps.binding.PS_ERR_INVALID


ALLOCATOR = r"""
#include <Python.h>
#include <c10/core/Allocator.h>
// forwards to the allocator it replaces and counts the allocations of at least `floor` bytes, and those made with the interpreter lock held
static c10::Allocator* before;
static size_t floor_bytes;
static int counted, held;
struct Counting : c10::Allocator {
    c10::DataPtr allocate(size_t n) override {
        if (n >= floor_bytes) ++counted, held += PyGILState_Check();
        return before->allocate(n);
    }
    c10::DeleterFnPtr raw_deleter() const override { return before->raw_deleter(); }
    void copy_data(void* d, const void* s, size_t n) const override { before->copy_data(d, s, n); }
};
extern "C" void install(long n) {
    static Counting mine;
    floor_bytes = (size_t)n;
    before = c10::GetAllocator(c10::DeviceType::CPU);
    c10::SetAllocator(c10::DeviceType::CPU, &mine, 100);
}
extern "C" int counts(int which) { return which ? held : counted; }
"""

ALLOCATE = """
import ctypes, sys
import torch
sys.path[:0] = %r
import test_tensor_calls_host as t
lib = ctypes.CDLL(%r)
pa = t.host_session()
pa._plan, pa._total_q, pa._n_q_heads, pa._ws_ptr, pa._ws_bytes = 0, 4096, 8, 0, 0
q, row = torch.zeros((4096, 8, 64), dtype=torch.bfloat16), torch.zeros((1, 256), dtype=torch.int32)
lib.install(4096 * 8 * 4)
for call in (lambda: pa.gather(row, 4096), lambda: pa.run(q, row)):
    try:
        call()
    except t.ps.PsError:
        pass
print(lib.counts(0), lib.counts(1))
"""


def test_results_are_allocated_without_the_interpreter_lock(tmp_path):
    """An allocation may wait for the device, and what it waits for may need the interpreter (a host function of a stream)."""
    src, so = tmp_path / "counting.cpp", str(tmp_path / "counting.so")
    src.write_text(ALLOCATOR)
    root = os.path.dirname(torch.__file__)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI), "-I",
                           os.path.join(root, "include"), "-I", sysconfig.get_paths()["include"], str(src), "-o", so, "-L", os.path.join(root, "lib"), "-lc10"])
    here = os.path.dirname(os.path.abspath(__file__))
    run = subprocess.run([sys.executable, "-c", ALLOCATE % ([here, os.path.dirname(here)], so)], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr
    assert run.stdout.split() == ["4", "0"]  # K and V, out and lse


def test_the_library_is_built_without_torch(tmp_path):
    """The C ABI and the planner need no torch, neither to be built nor to be loaded."""
    (tmp_path / "torch").mkdir()
    (tmp_path / "torch" / "__init__.py").write_text("raise ImportError('no torch here')\n")
    here = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    code = ("import sys; sys.path[:0] = [%r, %r]\nfrom paper_2507_17769_b200 import binding as B, build\nbuild.build_library()\n"
            "B.load(); assert 'torch' not in sys.modules\nassert not any('torch' in f for f in build.library_files())" % (str(tmp_path), here))
    run = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=300)
    assert run.returncode == 0, run.stderr


def test_the_extension_belongs_to_one_torch(monkeypatch):
    """Its file carries the version of torch that it was built against: another torch builds its own."""
    from paper_2507_17769_b200 import build

    here = build.torch_calls_path()
    monkeypatch.setattr(torch, "__version__", "1.2.3")
    assert build.torch_calls_path() != here and "1.2.3" in os.path.basename(build.torch_calls_path())


def test_without_the_extension_tensors_take_the_calls_through_addresses(monkeypatch):
    from paper_2507_17769_b200 import build

    monkeypatch.setattr(session, "_torch_calls", None)
    monkeypatch.setattr(build, "build_torch_calls", lambda *a, **k: (_ for _ in ()).throw(OSError("no compiler here")))
    with pytest.warns(RuntimeWarning, match="no compiler here"):
        assert session.torch_calls() is None
    assert session.torch_calls() is None  # (tried and told once)
    monkeypatch.setattr(session.PagedAttention, "__del__", lambda self: None)
    pa = host_session()
    session.take_tensors(pa)
    seen = []

    class Calls:
        def kv_write(self, *a):
            seen.append(a)
            return 0

    pa._calls = Calls()
    k, row = torch.zeros((1, 2, 64), dtype=torch.bfloat16), torch.zeros((1, 4), dtype=torch.int32)
    pa.write(k, k, row, [0], [1])
    assert seen[0][1:5] == (k.data_ptr(), k.data_ptr(), row.data_ptr(), 4)
