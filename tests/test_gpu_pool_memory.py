"""GPU: memory that live states keep between calls is bounded for all of them
together (1 GiB), and is given back when they go.

Sixteen states at chi = 1024 each run one two-site update through
apply_cluster / truncate_split, whose work buffers (theta twice, four 2048-wide
square matrices: 0.2 GiB and more) come from the state's pool and go back to it.
In use afterwards, per state: two sites of 16 MiB that are rewritten beside two
smaller ones, the direct solver's scratch and a MiB of staging, below 96 MiB
(products on the CUDA cores: the tensor cores' packed operands are scratch that a
state keeps by design)."""
import numpy as np
import pytest

from gpu_helpers import lib, random_unitary

pytestmark = pytest.mark.gpu

GIB = 1 << 30


def test_idle_memory_of_many_states_is_bounded():
    import torch
    P = lib()
    chi, count = 1024, 16
    chis = np.array([1, chi, chi, chi, 1], dtype=np.int32)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(3)
    sites = [torch.randn(a, 2, b, dtype=torch.complex64, device="cuda", generator=gen) / (2 * b) ** 0.5
             for a, b in zip(chis.tolist(), chis.tolist()[1:])]
    lams = [torch.full((c,), c ** -0.5, dtype=torch.float64, device="cuda") for c in chis.tolist()]
    U = random_unitary(4, np.random.default_rng(4))
    cfg = P.make_config(4, chi, 1e-8, 24, 0, 2, P.FP32)

    def update():
        mps = P.MPS(cfg)
        mps.load_device(chis, [x.data_ptr() for x in sites], [x.data_ptr() for x in lams])
        mps.apply_cluster(P.Cluster(1, 2, 0, 0), U)
        mps.truncate_split(P.Cluster(1, 2, 0, 0))
        return mps

    P.set_tensor_cores(0)
    try:
        _check(P, torch, update, count)
    finally:
        P.set_tensor_cores(1)


def _check(P, torch, update, count):
    update().close()                               # modules loaded, one-time memory taken
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    states = [update() for _ in range(count)]
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    print(f"{count} states hold {held / GIB:.2f} GiB")
    assert held <= GIB + count * 96 * (1 << 20)
    for m in states:
        m.close()
    torch.cuda.synchronize()
    left = before - torch.cuda.mem_get_info()[0]
    assert left <= 64 << 20
