"""The native half of the binding: what it refuses and how, without a device (the checks come before any launch)."""
import os
import subprocess
import sys
import sysconfig

import pytest
import torch

from paper_2409_09708_b200 import _elsa_host, binding as lib


def arguments(**changed):
    a = dict(X=torch.zeros(4, 64, dtype=torch.float16), vals=torch.zeros(8, 32, dtype=torch.float16), idx=torch.zeros(8, 3, dtype=torch.int32),
             bias=None, out=8, in_=64, N=4, M=8, code=0, Y=None, workspace=None, status=None, stream=0)
    a.update(changed)
    return list(a.values())


def test_arguments_of_the_wrong_kind():
    with pytest.raises(ValueError, match="contiguous"):
        _elsa_host.linear(*arguments(vals=torch.zeros(8, 64, dtype=torch.float16)[:, ::2]))
    with pytest.raises(TypeError, match="tensor expected"):
        _elsa_host.linear(*arguments(X=[1.0]))
    with pytest.raises(TypeError):
        _elsa_host.linear(*arguments(out="8"))
    with pytest.raises(TypeError, match="13 arguments"):
        _elsa_host.linear(*arguments()[:-1])
    with pytest.raises(IndexError):
        _elsa_host.compress(torch.zeros(64, dtype=torch.float16), 4, 8, 0, 0)
    with pytest.raises(ValueError, match="levels"):
        _elsa_host.compress_levels(torch.zeros(8, 64, dtype=torch.float16), (1, 2), 8, 0, 0)
    with pytest.raises(RuntimeError):
        _elsa_host.linear(*arguments(out=-8))


def test_a_status_of_the_entry_point_comes_back_as_a_number():
    assert _elsa_host.linear(*arguments(N=9)) == 3                     # ELSA_ERR_NM
    assert _elsa_host.compress(torch.zeros(8, 64, dtype=torch.float16), 9, 8, 0, 0) in (1, 3)
    with pytest.raises(lib.ElsaError) as e:
        lib._result(_elsa_host.linear(*arguments(M=5)))
    assert e.value.status == 3


class NullStream:
    cuda_stream = 0


def test_tensors_of_the_wrong_rank_are_refused():
    """A weight is [out, in] and a masked linear's activations [rows, in]; other ranks would be read as if the first two sizes were all."""
    f16 = lambda *shape: torch.zeros(shape, dtype=torch.float16)
    wrong = pytest.raises((ValueError, IndexError))
    for W in (f16(8, 4, 16), f16(1, 8, 64), f16(64)):
        with wrong:
            lib.elsa_nm_compress(W, 4, 8, stream=NullStream)
        with wrong:
            lib.elsa_nm_compress_levels(W, [1, 4], 8, stream=NullStream)
        with wrong:
            _elsa_host.compress_levels(W, [1, 4], 8, 0, 0)
        with wrong:
            lib.elsa_nm_linear_masked(f16(4, 64), W, None, 4, 8, stream=NullStream)
    for X in (f16(4, 2, 64), f16(64)):
        with wrong:
            lib.elsa_nm_linear_masked(X, f16(8, 64), None, 4, 8, stream=NullStream)


def test_the_module_is_of_this_python_and_torch(monkeypatch, tmp_path):
    from paper_2409_09708_b200 import build
    assert os.path.basename(_elsa_host.__file__) == "_elsa_host" + sysconfig.get_config_var("EXT_SUFFIX")
    assert _elsa_host.torch_version == torch.__version__
    stamp = tmp_path / "stamp"
    monkeypatch.setattr(build, "_older", lambda built, deps: False)     # what the sources' times say is another matter
    monkeypatch.setattr(build, "HOST_STAMP", str(stamp))
    assert build.host_is_stale()                                       # no record of a torch
    stamp.write_text("1.0")
    assert build.host_is_stale()
    stamp.write_text(torch.__version__)
    assert not build.host_is_stale()


@pytest.mark.parametrize("module", ["None", "type(sys)('paper_2409_09708_b200._elsa_host')"], ids=["missing", "other_torch"])
def test_a_module_that_does_not_fit_says_what_to_run(module):
    code = ("import sys, torch\nimport paper_2409_09708_b200 as p\nm = %s\nif m is not None: m.torch_version = '1.0'; p._elsa_host = m\n"
            "sys.modules['paper_2409_09708_b200._elsa_host'] = m\nimport paper_2409_09708_b200.binding" % module)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    run = subprocess.run([sys.executable, "-c", code], cwd=root, capture_output=True, text=True)
    assert run.returncode != 0 and "ImportError" in run.stderr and "python -m paper_2409_09708_b200.build" in run.stderr, run.stderr
