"""What the binding takes as arguments: whatever the Python conversions it stands for take."""
import pytest

import paper_1802_06058_b200 as vgc


def _layer(**changes):
    import torch
    x = torch.zeros(2, 4)
    d = {"is_conv": 0, "B": 2, "C": 4, "Cout": 4, "x_host": x, "delta_host": x, "x_dev": x, "delta_dev": x}
    d.update(changes)
    return d


class _Defaults(dict):                      # a mapping that makes missing keys up when they are asked for with []
    def __missing__(self, key):
        raise AssertionError(f"layer[{key!r}] asked for: an optional key has its default")


@pytest.mark.parametrize("layer", [_layer(is_conv=True), _layer(is_conv=0.0), _layer(is_conv="numpy"), _Defaults(_layer())])
def test_step_host_takes_layers_as_their_values_convert(layer):
    """is_conv is whatever int() takes, missing sizes are 1 (padding 0); the call gets as far as the staging buffers, which
    here are not on a GPU."""
    import numpy as np
    import torch
    if isinstance(layer["is_conv"], str):
        layer["is_conv"] = np.bool_(True)
    t = torch.zeros(16)
    with pytest.raises(TypeError, match="x_dev must be a CUDA tensor"):
        vgc.vgc_step_host([layer], t, t, t, t, t, torch.zeros(2, dtype=torch.int32), 2.0, 0.999, 1.0, None, t, t, None, None)


@pytest.mark.gpu
def test_scalars_are_whatever_float_takes():
    import numpy as np
    import torch
    x, d = torch.ones(2, 4, device="cuda"), torch.ones(2, 4, device="cuda")
    ws = torch.zeros(vgc.vgc_sqgrad_linear_workspace_bytes(2, 4, 4), dtype=torch.uint8, device="cuda")
    for scale in (1, 0.5, np.float32(0.5), np.float64(2), torch.tensor(0.25), "0.5", np.int64(3)):
        S = vgc.vgc_sqgrad_linear(x, d, scale, torch.zeros(16, device="cuda"), ws=ws)
        assert bool((S == 2 * float(scale)).all())
    with pytest.raises(ValueError):
        vgc.vgc_sqgrad_linear(x, d, "half", torch.zeros(16, device="cuda"), ws=ws)
