"""make_classes packs a fuel class as one record; the bytes are those of its
fields set one by one, also for classes with fields left out or values that
only float() or int() take, and what was refused is refused."""
import ctypes as C

import numpy as np
import pytest

import paper_1102_1343_gb300 as pkg
from paper_1102_1343_gb300 import synth


def field_by_field(classes):
    arr = (pkg.fire_fuel_class * len(classes))()
    for k, c in enumerate(classes):
        for name, typ in pkg.fire_fuel_class._fields_:
            val = c.get(name, 0)
            setattr(arr[k], name, int(val) if typ is C.c_int else float(val))
    return arr


@pytest.mark.parametrize("change", [
    {}, {"st": ...}, {"fgi": "0.25"}, {"chaparral": 1.0}, {"savr": np.float32(3.3)}, {"weight_is_tf": True},
    {"se": 3}, {"other": 5}, {"chaparral": "1"}, {"fgi": "x"}, {"fgi": None}, {"fgi": 1j}, {"chaparral": 2**40}])
def test_class_records(change):
    classes = [dict(c) for c in synth.random_classes(np.random.default_rng(0))]
    for name, v in change.items():
        if v is ...:
            del classes[3][name]
        else:
            classes[3][name] = v
    got = []
    for make in (field_by_field, pkg.make_classes):
        try:
            got.append(bytes(make(classes)))
        except Exception as e:  # noqa: BLE001
            got.append((type(e), str(e)))
    assert got[0] == got[1]
