"""The binding's structs hold the same bytes however a caller gives the
numbers: Python and numpy scalars, arrays and tensors, texts, values beyond
FP32, and states of fewer components (the rest zero)."""
import numpy as np
import pytest
import torch

import gen
from paper_2603_20525_gb300 import atp


@pytest.mark.parametrize("conv", [float, np.float64, np.float32, str, lambda v: torch.tensor(v, dtype=torch.float64),
                                  lambda v: np.float64(v).reshape(())])
def test_vehicle_and_cost(conv):
    for make, cls, d in ((atp.vehicle, atp.Vehicle, gen.vehicle_mrzr()), (atp.cost, atp.Cost, gen.cost_default(3, 4))):
        e = {k: conv(v) for k, v in d.items()}
        want = cls(**{k: float(e[k]) for k, _ in cls._fields_})
        assert bytes(make(dict(e, extra=1))) == bytes(want)
        with pytest.raises(KeyError):
            make({k: v for k, v in e.items() if k != "wt" and k != "M"})


def test_state():
    x = gen.uniform(1, 2, 13)
    want = bytes(atp.State(*[float(v) for v in x]))
    for y in (list(x), tuple(x), x, torch.as_tensor(x), iter(x), (str(v) for v in x)):
        assert bytes(atp.state(y)) == want
    assert bytes(atp.state(x[:7])) == bytes(atp.State(*[float(v) for v in x[:7]]))
    with pytest.raises(TypeError):
        atp.state(list(x) + [1.0])
    big = atp.state([1e40, float("nan")] + [0.0] * 11)
    assert np.isinf(big.x) and np.isnan(big.y)
