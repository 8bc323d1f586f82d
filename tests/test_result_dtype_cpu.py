"""Calls that write fp32 rows refuse a result of another type before anything is launched (no GPU: the library is a stand-in that must not
be reached)."""
import pytest
import torch

import paper_2505_18976_b200 as G
from paper_2505_18976_b200 import binding


@pytest.fixture
def calls(monkeypatch):
    """The calls on host tensors: device checks off, no compiled marshalling, a library that fails the test."""
    class NoMarshalling:
        def __getattr__(self, name):
            return lambda *a: None

    def reached():
        raise AssertionError("the library was reached")

    monkeypatch.setattr(binding, "_fast", NoMarshalling)
    monkeypatch.setattr(binding, "lib", reached)
    for name in ("_need_cuda", "_need_device_readable"):
        monkeypatch.setattr(binding, name, lambda *t: None)
    A, D = torch.zeros((2, 3, 8), dtype=torch.bfloat16), torch.zeros((2, 3, 6), dtype=torch.bfloat16)
    m = torch.arange(4, dtype=torch.int32)
    x, h = torch.zeros((2, 8)), torch.zeros((2, 8), dtype=torch.bfloat16)
    return {
        "factgrass_compress": (4, lambda out: G.factgrass_compress(A, D, m, m, 4, 1, 0, out=out)),
        "factgrass_compress_varlen": (4, lambda out: G.factgrass_compress_varlen(A, D, m, m, 4, 1, 0, 2, 3, out=out)),
        "grass_mask": (4, lambda out: G.grass_mask(x, m, out=out)),
        "factmask_compress": (16, lambda out: G.factmask_compress(A, D, m, m, out=out)),
        "grass_score": (2, lambda out: G.grass_score(x, x, out=out)),
        "grass_score_bf16": (2, lambda out: G.grass_score_bf16(h, h, out=out)),
    }


NAMES = ["factgrass_compress", "factgrass_compress_varlen", "grass_mask", "factmask_compress", "grass_score", "grass_score_bf16"]


@pytest.mark.parametrize("name", NAMES)
def test_result_of_another_type(calls, name):
    width, call = calls[name]
    for dtype in (torch.bfloat16, torch.float64, torch.int32):
        with pytest.raises(TypeError):
            call(torch.empty((2, width), dtype=dtype))


@pytest.mark.parametrize("name", NAMES)
def test_rows_that_are_not_contiguous(calls, name):
    width, call = calls[name]
    with pytest.raises(ValueError):
        call(torch.empty((width, 2)).t())


@pytest.mark.parametrize("name", NAMES)
def test_other_results_go_on_to_the_library(calls, name):
    width, call = calls[name]
    for out in (torch.empty((2, width)), torch.empty((3, width + 5))[1:, 2:2 + width]):
        with pytest.raises(AssertionError, match="the library was reached"):
            call(out)
