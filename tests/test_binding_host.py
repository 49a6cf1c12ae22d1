"""The binding's cache of C structs of shapes and rules (host only)."""
import dataclasses

import pytest

from paper_2609_27373_gb300 import wise

SHAPE = wise.Shape(1, 256, 2, 2, 64, 64, 0.0)
SELECT = wise.Select(1, 1, wise.WISE_SEL_TOPK, 2, 0.5, 4)


def _struct(value):
    return wise._c(value) if isinstance(value, wise.Shape) else wise._c_select(value)


@pytest.mark.parametrize("value", [SHAPE, SELECT])
def test_an_equal_value_of_a_refused_type_is_refused(value):
    _struct(value)  # the struct of the valid value is cached
    for f in dataclasses.fields(value):
        v = getattr(value, f.name)
        if isinstance(v, int):
            other = dataclasses.replace(value, **{f.name: float(v)})
            assert other == value
            with pytest.raises(TypeError):
                _struct(other)


def test_structs_hold_the_values():
    for value in (SHAPE, SELECT, dataclasses.replace(SHAPE, scale=1, batch=3), dataclasses.replace(SHAPE, scale=1.0, batch=3)):
        got = _struct(value)._obj
        assert bytes(got) == bytes(value.c())
        assert bytes(_struct(dataclasses.replace(value))._obj) == bytes(got)
    assert _struct(dataclasses.replace(SHAPE))._obj is _struct(SHAPE)._obj  # an equal value: the same struct
