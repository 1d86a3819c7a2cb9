"""The native module of the per-step calls is tied to the torch it was built with; the library is not."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_2411_04975_b200 import binding, build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def package(tmp_path):
    """A copy of the built package whose native module is of another torch: a file that does not load."""
    build.build()
    shutil.copytree(os.path.join(ROOT, "include"), tmp_path / "include")
    pkg = tmp_path / "paper_2411_04975_b200"
    shutil.copytree(os.path.join(ROOT, "paper_2411_04975_b200"), pkg, ignore=shutil.ignore_patterns("_call*.so", "__pycache__"))
    for name in ("_call.so", "_call.cpython-312-torch-0.0.1.so"):
        (pkg / name).write_bytes(b"of another torch")
    return tmp_path


def _run(where, code, **env):
    return subprocess.run([sys.executable, "-c", code], cwd=where, env=dict(os.environ, PYTHONPATH=str(where), **env), capture_output=True,
                          text=True, timeout=300)


def test_library_loads_without_a_module_for_this_torch(package):
    """No compiler either: the library still loads, the calls' arguments are converted in Python."""
    p = _run(package, """
import warnings
warnings.simplefilter("error")
import paper_2411_04975_b200 as sfx
from paper_2411_04975_b200 import binding
try:
    sfx.library()
except RuntimeWarning as e:
    print("warned:", e)
warnings.simplefilter("ignore")
sfx.library().sd_free(None)
print(type(binding._loaded()).__name__)
import torch
t = torch.zeros(2, dtype=torch.int32)
for call in (lambda: sfx.sd_append(None, t, t, t), lambda: sfx.sd_speculate(None, t, 4, 1.0, 4, 0, None, {})):
    try:
        call()
    except TypeError as e:
        print(e)
""", PATH="/nonexistent")
    assert p.returncode == 0, p.stderr[-2000:]
    out = p.stdout.splitlines()
    assert out[0].startswith("warned: the native module of the per-step calls could not be had") and out[1] == "_PlainCall"
    assert out[2:] == ["slots: expected a contiguous CUDA (or pinned host) tensor of torch.int32, got torch.int32 on cpu"] * 2


def test_module_is_built_for_the_torch_that_is_there(package):
    p = _run(package, """
import torch
torch.__version__ = "99.1"
from paper_2411_04975_b200 import binding, build
asked = []
def build_call():
    asked.append(build.call_path())
    raise OSError("enough")
build.build_call = build_call
binding.library()
print(asked)
""")
    assert p.returncode == 0, p.stderr[-2000:]
    assert "torch-99.1.so" in p.stdout


def test_plain_calls_take_the_same_arguments():
    """The two forms of each call agree on the number of arguments (the native one counts them)."""
    import inspect
    binding.library()
    native = binding._load_call(binding._lib)
    for name in ("speculate", "step", "append"):
        n = len(inspect.signature(getattr(binding._PlainCall(binding._lib), name)).parameters)
        with pytest.raises(TypeError, match=f"{n} arguments expected"):
            getattr(native, name)()
