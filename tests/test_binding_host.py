"""What the Python binding accepts, refuses and hands on before a kernel runs (no GPU needed: the calls that go through
reach the library with a null context, which it refuses as a bad argument)."""
import ctypes as C

import numpy as np
import pytest
import torch

import paper_2605_04478_b200 as ccld
from helpers import make_cols
from paper_2605_04478_b200.build import build


@pytest.fixture(scope="module")
def an():
    """An analyzer without a context."""
    build()
    a = ccld.Analyzer.__new__(ccld.Analyzer)
    a.lib, a.torch, a.h, a._keep, a._n_comms = ccld.load_library(), torch, C.c_void_p(), {}, 0
    return a


def columns(n=4):
    return make_cols(dict(rank=i, seq=0, t_enter=1000 + i, t_exit=2000 + i) for i in range(n))


def refused_by_the_library(call):
    with pytest.raises(ccld.CcldError) as e:
        call()
    assert e.value.code == -1


@pytest.mark.parametrize("missing", ["absent", "none", "misspelt"])
@pytest.mark.parametrize("general", [False, True])
def test_upload_without_ranks_is_refused(an, missing, general):
    """Both ways in: plain numpy columns, and the general way (a column that is a tensor)."""
    cols = columns()
    if general:
        cols["t_enter"] = torch.from_numpy(cols["t_enter"])
    refused_by_the_library(lambda: an.trace_upload(0, cols))
    rank = cols.pop("rank")
    if missing == "none":
        cols["rank"] = None
    elif missing == "misspelt":
        cols["ranks"] = rank
    with pytest.raises(ValueError):
        an.trace_upload(0, cols)
    assert not an._keep


@pytest.mark.parametrize("general", [False, True])
@pytest.mark.parametrize("name", ["bytes", "t_enter", "t_exit"])
def test_upload_of_object_columns_is_refused(an, name, general):
    """An array of Python objects has entries of eight bytes too: their addresses are no column."""
    cols = columns()
    cols[name] = np.array([int(v) for v in cols[name]], dtype=object)
    if general:
        cols["rank"] = torch.from_numpy(cols["rank"].view(np.int32))
    with pytest.raises(TypeError):
        an.trace_upload(0, cols)


@pytest.mark.parametrize("name,view", [("rank", "i4"), ("comm", "f4"), ("seq", ">u4"), ("bytes", "f8"), ("t_enter", "M8[ns]"), ("t_exit", "u8"), ("op", "?")])
def test_upload_takes_columns_by_their_bits(an, name, view):
    """Plain arrays of another type of the column's size go through as they are."""
    cols = columns()
    cols[name] = cols[name].view(view)
    refused_by_the_library(lambda: an.trace_upload(0, cols))


def test_capacities_beyond_any_list(an):
    """Room is taken for what the library can list, not for what the caller could hold: no capacity takes the process down."""
    for cap in (0, -5, 1 << 33, 1 << 62, (1 << 63) - 1):
        refused_by_the_library(lambda: an.locate_hang(0, 0, 0, roots_cap=cap))
        refused_by_the_library(lambda: an.opset_check(0, 0, 0, ranks_cap=cap))
        refused_by_the_library(lambda: an.locate_hangs(0, cap=cap))
        refused_by_the_library(lambda: an.locate_hangs(0, roots_stride=cap))
        refused_by_the_library(lambda: an.locate_hangs(0, cap=cap, roots_stride=cap))
