"""The memory per time step that the header states for a group of the NLL and
gradient (max_group_steps), where the leaf length changes with the size."""
import os
import re

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_00426_gb300 import workloads as W

HEADER = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "include",
                      "sqsm.h")


def _stated():
    """{(dtype, largest steps or None): KB} from the option's comment."""
    text = open(HEADER).read()
    text = text[text.index("max_group_steps;"):text.index("} sqsm_options;")]
    text = re.sub(r"\s+", " ", text)
    f32, f64 = text.split("KB in FP32", 1)[0], text.split("in FP64,", 1)[1]
    big = float(re.findall(r"([\d.]+)\s*$", f32)[0])
    small, upto = re.search(r"\(([\d.]+) KB in groups of up to (\d+) steps\)", text).groups()
    d = {(torch.float32, None): big, (torch.float32, int(upto)): float(small)}
    for kb, n in re.findall(r"([\d.]+) KB up to (\d+)", f64):
        d[(torch.float64, int(n))] = float(kb)
    d[(torch.float64, None)] = float(re.search(r"and ([\d.]+) KB above", f64).group(1))
    return d


@pytest.mark.parametrize("dtype,lengths,upto", [
    (torch.float32, [1000] * 16, 116_736), (torch.float32, [65_537], 116_736),
    (torch.float32, [120_000], None), (torch.float32, [400_000], None),
    (torch.float64, [8192], 16_384), (torch.float64, [16_384], 16_384),
    (torch.float64, [1000] * 16, 16_384), (torch.float64, [16_385], 65_536),
    (torch.float64, [65_536], 65_536), (torch.float64, [1000] * 64, 65_536),
    (torch.float64, [65_537], 116_736), (torch.float64, [116_736], 116_736),
    (torch.float64, [120_000], None), (torch.float64, [100_000] * 4, None)])
def test_memory_per_step_is_within_the_stated(dtype, lengths, upto):
    from paper_2207_00426_gb300 import binding as B
    kb = _stated()[(dtype, upto)]
    n, nb = sum(lengths), len(lengths)
    f64 = torch.float64

    def new(*shape, dt=dtype):
        return torch.zeros(shape, dtype=dt, device="cuda:0")

    y, m0 = new(n, 2), new(nb, 5) + 0.1
    N0 = 0.1 * torch.eye(5, dtype=dtype, device="cuda:0").repeat(nb, 1, 1)
    out = dict(ms=new(n + nb, 5), Ns=new(n + nb, 5, 5), nll=new(1, dt=f64), grad=new(3, dt=f64),
               change=new(1, dt=f64))
    off = np.concatenate([[0], np.cumsum(lengths)])
    # (the device code of a first call is loaded before the reading)
    first = B.Context(0, use_graph=False)
    B.sqsm_ipls_nll_grad(first, W.CT_THETA_TRUE, y[:10], [0, 10], m0[:1], N0[:1], 1, 1)
    torch.cuda.synchronize()
    first.close()
    ctx = B.Context(0, use_graph=False)
    free0 = torch.cuda.mem_get_info()[0]
    B.sqsm_ipls_nll_grad(ctx, W.CT_THETA_TRUE, y, off, m0, N0, 1, 1, **out)
    torch.cuda.synchronize()
    per_step = (free0 - torch.cuda.mem_get_info()[0]) / n
    ctx.close()
    print(per_step)
    # device memory is taken in units of 2 MiB
    assert 0.8 * 1000 * kb <= per_step <= 1000 * kb + 2 * 2 ** 20 / n
