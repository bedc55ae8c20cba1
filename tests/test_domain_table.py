"""The domain records that reach the library, filled column by column, against one
assignment per number."""
import ctypes
from types import SimpleNamespace as D

import numpy as np
import pytest

from paper_1407_2052_gb300 import amrfd as A


def _plain(domains):
    arr = (A.DomainC * len(domains))()
    for c, d in zip(arr, domains):
        for k in range(3):
            c.n[k], c.nb[k], c.dx[k] = int(d.n[k]), int(d.nb[k]), float(d.dx[k])
            for f in range(2):
                c.bc[k][f] = int(d.bc[k][f])
                if getattr(d, "asym", None) is not None:
                    c.asym[k][f] = int(d.asym[k][f])
        c.offset = int(d.offset)
    return arr


BC = ((0, 0), (1, 1), (2, 1))
CASES = {
    "empty": [],
    "one": [D(n=(5, 6, 7), nb=(5, 2, 1), dx=(0.1, 0.2, 0.3), bc=BC, offset=11)],
    "shared_and_distinct": [D(n=(8, 8, 4 + i % 3), nb=(2, 1, 1), dx=(0.5, 1.0 / (i + 1), 2), bc=BC, offset=i << 33,
                              asym=((1, 2), (0, 0x80000000), (3, i)) if i % 2 else None) for i in range(9)],
    "lists_arrays_and_longer": [
        D(n=[4, 5, 6], nb=np.array([1, 5, 2]), dx=np.array([0.1, 0.2, 0.3]), bc=[[0, 0], [1, 2], [2, 2]], offset=0),
        D(n=(4.0, np.int32(5), True), nb=(1, 1, 1, 9), dx=[1, 2, 3], bc=np.zeros((3, 2)), offset=np.int64(7),
          asym=[[1, 0], [0, 1], [0, 0]])],
}


@pytest.mark.parametrize("name", CASES)
def test_domain_records(name):
    want, got = _plain(CASES[name]), A.domains_c(CASES[name])
    assert len(got) == len(want) and ctypes.sizeof(got) == ctypes.sizeof(want)
    assert bytes(got) == bytes(want)


@pytest.mark.parametrize("field", ["n", "nb", "dx", "bc"])
def test_short_fields_stay_refused(field):
    d = dict(n=(5, 6, 7), nb=(5, 2, 1), dx=(0.1, 0.2, 0.3), bc=BC, offset=0)
    d[field] = d[field][:1]
    with pytest.raises(IndexError):
        A.domains_c([D(**d), D(**d)])


@pytest.mark.parametrize("field,value", [("n", (2 ** 32 + 16, 16, 1)), ("nb", (2 ** 32 + 1, 1, 1)),
                                         ("n", (2 ** 31 + 8, 2 ** 31, 2 ** 31))])
def test_sizes_beyond_the_records_types_are_not_taken_for_small_ones(field, value):
    """The time step of many blocks sizes its tensors from the numbers given, not from what a
    record of 32-bit sizes holds of them."""
    torch = pytest.importorskip("torch")
    d = dict(n=(16, 16, 1), nb=(1, 1, 1), dx=(1.0, 1.0, 1.0), bc=((0, 0),) * 3, offset=0)
    d[field] = value
    U, out, act = torch.zeros(9 * 256, dtype=torch.float64), torch.zeros(1, dtype=torch.float64), torch.ones(1, dtype=torch.uint8)
    with pytest.raises(ValueError):
        A.dt_noalloc(A.MHD_GLM, 2, 1.4, 0.4, [D(**d)], U, out, active=act if field == "nb" else None)


def test_a_missing_spacing_stays_refused():
    d = D(n=(5, 6, 7), nb=(1, 1, 1), dx=(0.1, None, 0.3), bc=BC, offset=0)
    with pytest.raises(TypeError):
        A.domains_c([d])
    d.dx = (0.1, float("nan"), 0.3)
    assert np.isnan(A.domains_c([d])[0].dx[1])


@pytest.mark.parametrize("name", [c for c in CASES if CASES[c]])
@pytest.mark.parametrize("few", [0, 100], ids=["table", "one_by_one"])
def test_both_ways_of_filling_give_the_same_records(few, name, monkeypatch):
    monkeypatch.setattr(A, "_FEW", few)
    doms = CASES[name]
    arr, nblocks, need = A._domain_records(doms, 9)
    assert bytes(arr) == bytes(_plain(doms))
    assert nblocks == sum(int(d.nb[0]) * int(d.nb[1]) * int(d.nb[2]) for d in doms)
    assert need == max(int(d.offset) + 9 * int(d.n[0]) * int(d.n[1]) * int(d.n[2]) for d in doms)


@pytest.mark.parametrize("few", [0, 100], ids=["table", "one_by_one"])
@pytest.mark.parametrize("field,value", [("n", (2 ** 32 + 16, 16, 1)), ("nb", (2 ** 32 + 1, 1, 1))])
def test_both_ways_refuse_sizes_beyond_the_records_types(few, field, value, monkeypatch):
    monkeypatch.setattr(A, "_FEW", few)
    test_sizes_beyond_the_records_types_are_not_taken_for_small_ones(field, value)
