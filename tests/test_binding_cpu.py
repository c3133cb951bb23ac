"""Host logic of the Python binding that needs no GPU: the marshalling of a
batch of problems into the device addresses and lengths that
dpd_estimate_batched takes.  The tensor checks (complex64, CUDA, contiguous)
are replaced by a no-op so that CPU tensors stand in for device ones; the
address arithmetic is the same."""
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import paper_1612_09001_gb300 as dpd

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture
def cpu_tensors_allowed(monkeypatch):
    monkeypatch.setattr(dpd, "_check_samples", lambda t, name: None)


def test_two_d_batch_gives_row_addresses(cpu_tensors_allowed):
    X = torch.zeros((5, 12), dtype=torch.complex64)
    addr, lens, dev = dpd._batch_pointers(X, "u")
    assert addr.dtype == np.uint64 and lens.dtype == np.int64
    assert [int(a) for a in addr] == [X.data_ptr() + 12 * 8 * i for i in range(5)]
    assert [int(n) for n in lens] == [12] * 5
    assert dev == X.device


def test_list_of_rows_matches_the_two_d_form(cpu_tensors_allowed):
    X = torch.zeros((4, 7), dtype=torch.complex64)
    a2, n2, _ = dpd._batch_pointers(X, "u")
    al, nl, _ = dpd._batch_pointers(list(X), "u")
    assert np.array_equal(a2, al) and np.array_equal(n2, nl)


def test_list_of_different_lengths(cpu_tensors_allowed):
    xs = [torch.zeros(n, dtype=torch.complex64) for n in (3, 1, 9)]
    addr, lens, _ = dpd._batch_pointers(xs, "u")
    assert [int(a) for a in addr] == [x.data_ptr() for x in xs]
    assert [int(n) for n in lens] == [3, 1, 9]


@pytest.mark.parametrize("bad", [torch.zeros(6, dtype=torch.complex64),            # 1-D tensor
                                 torch.zeros((0, 4), dtype=torch.complex64),       # no problems
                                 torch.zeros((3, 0), dtype=torch.complex64),       # empty rows
                                 torch.zeros((2, 2, 2), dtype=torch.complex64)])   # 3-D
def test_malformed_batches_are_refused(cpu_tensors_allowed, bad):
    with pytest.raises(ValueError):
        dpd._batch_pointers(bad, "u")


def test_empty_list_is_refused(cpu_tensors_allowed):
    with pytest.raises(ValueError):
        dpd._batch_pointers([], "u")


def test_checks_still_run_without_the_stand_in():
    """With the real checks a CPU tensor (not a CUDA one) is refused before any
    address is formed, in both forms."""
    X = torch.zeros((2, 4), dtype=torch.complex64)
    with pytest.raises(ValueError):
        dpd._batch_pointers(X, "u")
    with pytest.raises(ValueError):
        dpd._batch_pointers(list(X), "u")
    with pytest.raises(TypeError):
        dpd._batch_pointers([torch.zeros(4, dtype=torch.float32)], "u")


def test_current_stream_without_torchs_private_names(monkeypatch):
    """A torch without the private accessors: the public current stream serves."""
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.delattr(torch._C, name, raising=False)
    for name in ("_empty_like", "_raw_stream", "_current_device"):
        monkeypatch.setattr(dpd, name, None)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device: type("S", (), {"cuda_stream": 1000 + device}))
    assert dpd._stream_ptr(None) == 1003
    assert dpd._stream_ptr(type("S", (), {"cuda_stream": 7})) == 7


def test_direct_learning_imports_without_torchs_private_hook_lists():
    code = ("import importlib; o = importlib.import_module('torch.optim.optimizer'); "
            "del o._global_optimizer_pre_hooks, o._global_optimizer_post_hooks; import paper_1612_09001_gb300.direct")
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, cwd=ROOT)
    assert r.returncode == 0, r.stderr


def test_direct_learning_steps_without_the_optimizer_submodules_name(monkeypatch):
    """Versions of torch whose torch.optim does not keep the name of its submodule: the step
    still tells a plain optimiser from a hooked one (here: no state yet, torch's own step)."""
    from paper_1612_09001_gb300.direct import DirectLearner
    monkeypatch.delattr(torch.optim, "optimizer", raising=False)
    lr = DirectLearner.__new__(DirectLearner)
    lr.param = torch.nn.Parameter(torch.ones(3))
    lr.param.grad = torch.ones(3)
    lr.opt = torch.optim.Adam([lr.param], lr=0.1)
    lr._adam_step()
    assert torch.allclose(lr.param.detach(), torch.full((3,), 0.9), atol=1e-6)
