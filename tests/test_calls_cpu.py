"""The two ways the per-step calls are marshalled (the C extension, and ctypes where it cannot be compiled) check and pass the
same arguments.  No GPU: every call here is refused before anything is launched."""
import subprocess

import pytest
import torch

import paper_2411_10666_b200.binding as binding


class _Stream:
    cuda_stream = 0


@pytest.fixture(params=["extension", "no compiler", "no headers", "not loadable"])
def marshalling(request, monkeypatch):
    monkeypatch.setattr(binding, "_calls", None)
    monkeypatch.setattr(binding, "_fn", {})
    if request.param == "extension":
        return request.param

    def build_calls(force=False):
        if request.param == "no compiler":
            raise FileNotFoundError("gcc")
        if request.param == "no headers":
            raise subprocess.CalledProcessError(1, "gcc")
        return __file__                                     # a file that is no extension module

    monkeypatch.setattr(binding._build, "build_calls", build_calls)
    with pytest.warns(RuntimeWarning, match="ctypes"):
        binding._hot("sam_step")
    return request.param


def _refusals(call, *args):
    try:
        call(*args, stream=_Stream)
    except (binding.SamError, TypeError, AssertionError) as e:
        return type(e), getattr(e, "code", None)
    raise AssertionError("accepted")


def test_null_handles_are_refused_by_the_library(marshalling):
    none6 = (None,) * 6
    arg = (binding.SamError, -1)
    assert _refusals(binding.sam_step, None, None, 4, None, 4, *none6) == arg
    assert _refusals(binding.sam_step_host, None, None, 4, None, 4, *none6) == arg
    draft = torch.zeros(2, 4, dtype=torch.int32)
    assert _refusals(binding.sam_step_host, None, draft, 4, draft[0], 4, *none6) == arg        # host tensors are what it takes


def test_host_tensors_where_the_gpu_reads_are_type_errors(marshalling):
    i, f = torch.zeros(2, 4, dtype=torch.int32), torch.zeros(2, 4)
    n = torch.zeros(2, dtype=torch.int32)
    bad = (TypeError, None)
    assert _refusals(binding.sam_step, None, i, 4, n, 4, i, n, i, n, i, n) == bad
    assert _refusals(binding.sam_step_verified, None, i, i, n, None, 4, i, n, i, n, i, n) == bad
    assert _refusals(binding.sam_accept_greedy, i, n, i, None, i, n) == bad
    assert _refusals(binding.sam_select_auxiliary, i, n, n, i, n) == bad
    assert _refusals(binding.sam_tree_draft, None, n, n, 4, 1, i, i, f, n) == bad
    assert _refusals(binding.sam_retrieve_noalloc, None, 9, i, n, 4, 0, 1, i, n, i, n, i, n) == bad
    m, fn = binding._hot("sam_step")

    class Out:
        draft_tokens, draft_len, match_len, source, state, status = i, n, i, n, i, n

        def tensors(self):
            return (i, n, i, n, i, n)

    with pytest.raises(TypeError):
        m.step_out(fn, 0, i, n, 4, Out(), 0)


def test_host_arrays_of_the_wrong_type_are_refused(marshalling):
    f, n = torch.zeros(2, 4), torch.zeros(2, dtype=torch.int32)
    kind, _ = _refusals(binding.sam_step_host, None, f, 4, n, 4, n, n, n, n, n, n)
    assert kind in (TypeError, AssertionError)
