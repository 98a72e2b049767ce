"""The Python entry points as names of the package: star import, pickles, a tree that is not built, and arguments that
are refused before anything reaches the device.  No GPU needed."""
import os
import pickle
import shutil
import subprocess
import sys
import sysconfig
from unittest.mock import Mock

import pytest
import torch

import paper_1804_08066_b200 as mqg

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _python(code, cwd=ROOT, **env):
    out = subprocess.run([sys.executable, "-c", code], cwd=cwd, capture_output=True, text=True, timeout=300,
                         env={**os.environ, **env})
    assert out.returncode == 0, out.stderr[-2000:]
    return out.stdout


def test_star_import_brings_every_entry_point():
    out = _python("from paper_1804_08066_b200 import *\n"
                  "import paper_1804_08066_b200 as m\n"
                  "print(len(m._NATIVE), sorted(n for n in m._NATIVE if n not in globals()), 'mqg_code_words' in globals())")
    assert out.split(None, 1) == ["18", "[] True\n"]


def test_entry_points_pickle_by_the_package_s_name():
    data = pickle.dumps([mqg.mqg_quantize, mqg.mqg_server_step])
    assert pickle.loads(data) == [mqg.mqg_quantize, mqg.mqg_server_step]
    # and in a process that has loaded nothing yet
    assert "mqg_server_step" in _python("import pickle; print(pickle.loads(%r))" % data)


def test_names_exist_where_nothing_is_built(tmp_path):
    pkg = tmp_path / "paper_1804_08066_b200"
    shutil.copytree(os.path.join(ROOT, "paper_1804_08066_b200"), pkg,
                    ignore=shutil.ignore_patterns("*.so", "csrc", "__pycache__"))
    out = _python("from paper_1804_08066_b200 import *\n"
                  "import paper_1804_08066_b200 as m\n"
                  "assert hasattr(m, 'mqg_quantize') and mqg_quantize.__name__ == 'mqg_quantize'\n"
                  "try:\n"
                  "    mqg_quantize(None, 0, 4, 32, 0, None, None)\n"
                  "except ImportError as e:\n"
                  "    print(e)", cwd=tmp_path)
    assert "is not built" in out


NO_HEAP = r"""
#include <cstdlib>
#include <new>
extern "C" { int no_heap = 0; }
void* operator new(std::size_t n)
{
    void* p = no_heap ? nullptr : std::malloc(n ? n : 1);
    if (!p) throw std::bad_alloc();
    return p;
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
"""


def test_no_exception_leaves_the_c_abi(tmp_path):
    """The calls that take segment tables need no memory of the host's heap, however many segments there are."""
    (tmp_path / "no_heap.cpp").write_text(NO_HEAP)
    lib = str(tmp_path / "no_heap.so")
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", str(tmp_path / "no_heap.cpp"), "-o", lib], check=True)
    out = _python("""
import ctypes as C
import paper_1804_08066_b200 as mqg
lib, no_heap = mqg.raw_library(), C.c_int.in_dll(C.CDLL(%r), "no_heap")
nseg = 300
off = (C.c_uint64 * (nseg + 1))(*[65536 * j for j in range(nseg + 1)])       # long segments, all aligned
p = C.c_void_p(0x10000)                                                      # never dereferenced on the host
tab = (C.c_void_p * 2)(0x10000, 0x20000)
quantize = lambda: lib.mqg_quantize_segments_workers(tab, 2, nseg, off, off, 4, 0, tab, tab, 0, 0, 0, 0, None)
server = lambda: lib.mqg_server_step_segments(tab, tab, 2, 4, nseg, off, off, p, 0.1, None, None)
st = [quantize(), server()]                                                  # what the first call sets up is done
no_heap.value = 1
st += [quantize(), server()]
no_heap.value = 0
print(st)
""" % lib, LD_PRELOAD=lib, CUDA_VISIBLE_DEVICES="")                              # no device: no launch, on any machine
    assert out.strip() == str([mqg.MQG_ERR_CUDA] * 4)


def test_objects_that_only_look_like_tensors_are_refused():
    like = Mock(spec=torch.Tensor)
    assert isinstance(like, torch.Tensor)
    for call in (lambda: mqg.mqg_apply(like, like, 0.1, 4),
                 lambda: mqg.mqg_quantize(like, 0, 4, 32, 0, None, None),
                 lambda: mqg.mqg_server_step([like], [like], 1, 4, 32, 32, like, 0.1)):
        with pytest.raises(TypeError, match="tensor"):
            call()


class Shrinking:
    """A number whose conversion empties the list it stands in."""

    def __init__(self, home):
        self.home = home

    def __int__(self):
        self.home.clear()
        return 0

    __index__ = __int__


def test_a_list_that_changes_while_it_is_read():
    offsets = []
    offsets += [Shrinking(offsets)] + [10**6 * j for j in range(1, 60)]
    with pytest.raises(TypeError, match="grad must be a CUDA tensor"):
        mqg.mqg_quantize_segments(None, offsets, list(range(60)), 4, 0, None, None)
    assert not offsets


def test_what_empty_lists_of_workers_raise():
    with pytest.raises(TypeError, match="same dtype"):
        mqg.mqg_quantize_workers([], 0, 0, 4, 32, 0, [], [])
    with pytest.raises(TypeError, match="same dtype"):
        mqg.mqg_quantize_workers_minmax([], 0, 0, 4, 32, [], [])
    with pytest.raises(IndexError):
        mqg.mqg_quantize_segments_workers([], 0, [0], [0], 4, 0, [], [])


def test_the_binding_fits_one_interpreter_and_one_torch(monkeypatch):
    from paper_1804_08066_b200 import build
    here = build.binding_path()
    assert os.path.exists(here) and here.endswith(sysconfig.get_config_var("EXT_SUFFIX"))
    assert mqg.mqg_quantize.__self__.__file__ == here
    monkeypatch.setattr(torch, "__version__", "9.8.7")
    assert "9.8.7" in build.binding_path() and not os.path.exists(build.binding_path())
    out = _python("import torch\n"
                  "torch.__version__ = '9.8.7'\n"
                  "import paper_1804_08066_b200 as m\n"
                  "try:\n"
                  "    m.mqg_quantize(None, 0, 4, 32, 0, None, None)\n"
                  "except ImportError as e:\n"
                  "    print(e)")
    assert "9.8.7" in out and "is not built" in out
