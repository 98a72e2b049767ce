"""The Python entry points as names of the package: star import, pickles, a tree that is not built, and arguments that
are refused before anything reaches the device.  No GPU needed."""
import os
import pickle
import shutil
import subprocess
import sys

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
