"""The binding's pointer array of E expert matrices (`_ptrs`): one contiguous [E x ...] tensor takes a
base address and E steps; every form it accepts must give what slicing and `_ptr` give, and what was
refused stays refused. CPU tensors posing as CUDA ones: no launch happens here."""
import pytest
import torch

from paper_2606_28516_gb300 import clearmoe as cm


class Posing:
    """A CPU tensor that says it is on the GPU (as do its slices)."""

    is_cuda = True

    def __init__(self, t):
        self.t = t

    def __getitem__(self, i):
        return Posing(self.t[i])

    def __len__(self):
        return len(self.t)

    def __getattr__(self, name):
        return getattr(self.t, name)


def _general(ts, E):
    return [cm._ptr(ts[e]) for e in range(E)]


BASE = torch.arange(12 * 8 * 16, dtype=torch.float32)


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("form", ["whole", "first", "offset", "outer_stride", "one", "one_strided", "inner_one", "list"])
def test_same_pointers_as_slicing(form, dtype):
    t = BASE.to(dtype).reshape(12, 8, 16)
    E = {"first": 5, "outer_stride": 6, "one": 1, "one_strided": 1}.get(form, 12)
    if form == "offset":
        t, E = t[3:], 9
    elif form == "outer_stride":
        t = t[::2]  # every matrix contiguous, the whole not
    elif form == "one_strided":
        t = t[4:5].as_strided((1, 8, 16), (7, 16, 1), t[4:5].storage_offset())  # a size-1 dimension: any stride
    elif form == "inner_one":
        t = t.reshape(12, 128, 1)
    p = [Posing(v) for v in t] if form == "list" else Posing(t)
    assert list(cm._ptrs(p, E)) == _general(p, E)


def test_refused_forms_stay_refused():
    t = BASE.reshape(12, 8, 16)
    with pytest.raises(ValueError):
        cm._ptrs(t, 12)  # not on the GPU
    with pytest.raises(ValueError):
        cm._ptrs(Posing(t.transpose(1, 2)), 12)  # matrices not contiguous
    with pytest.raises(IndexError):
        cm._ptrs(Posing(t), 13)  # fewer matrices than experts
    with pytest.raises(ValueError):
        cm._ptrs([Posing(t[0]), t[1]], 2)
