"""Shared memory of a launch: set counts whose tile prefix comes close to what a
kernel gets without opting in, and threads that launch one kernel with
different sizes at the same time."""
import math
import threading

import numpy as np
import pytest

from paper_2307_04843_gb300 import workloads

L = 2 * math.pi


@pytest.mark.gpu
@pytest.mark.parametrize("n_sets", [600, 1000, 1300, 1700, 1800, 4096])
@pytest.mark.parametrize("kind", ["flying", "gauss"])
def test_batched_push_at_every_set_count(kind, n_sets):
    """With a node grid a block of 128 holds 34 KB besides the prefix; the static
    part (pulse, component table) counts against the same 48 KB."""
    import torch
    from paper_2307_04843_gb300 import _lib
    pulse = dict(kind=kind, pol="x", a0=1.0, omega=1.0, w0=2.5 * L)
    pulse.update(dict(env="cw", n_comp=2, bw_frac=0.05, beta_f=0.9, ff_length=20 * L) if kind == "flying"
                 else dict(env="gauss", env_len=25.0))
    box = ((-4 * L, 4 * L),) * 3
    lo, hi = (-4 * L,) * 3, (4 * L,) * 3
    g = torch.as_tensor(workloads.grid_field(box, 8, amplitude=0.2)).cuda()
    parts = workloads.particles_uniform(box, n_sets, 2)
    off = torch.arange(n_sets + 1, dtype=torch.int64, device="cuda")
    res = []
    with _lib.Handle([pulse] * n_sets) as h:
        ws = torch.zeros(64, dtype=torch.int32, device="cuda")
        dev = _lib.to_device(parts, "fp32")
        _lib.ap_gather_push_batched(h.h, dev, off, (g, lo, hi), -3.0, 0.02, 5, "fp32", None, ws)
        assert h.status() == 0
        res.append(_lib.to_host(dev))
    with _lib.Handle(pulse) as h:
        dev = _lib.to_device(parts, "fp32")
        h.push(dev, -3.0, 0.02, 5, precision="fp32", grid=(g, lo, hi))
        res.append(_lib.to_host(dev))
    for k in res[0]:
        np.testing.assert_array_equal(res[0][k], res[1][k], err_msg=k)


@pytest.mark.gpu
def test_threads_launch_one_kernel_with_different_sizes():
    import torch
    from paper_2307_04843_gb300 import _lib
    pulse = dict(kind="gauss", pol="x", a0=1.0, omega=1.0, w0=2.5 * L, env="gauss", env_len=25.0)
    errors = []
    start = threading.Barrier(2)

    def work(n_sets):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream), _lib.Handle([pulse] * n_sets) as h:
                parts = _lib.to_device(workloads.particles_uniform(((-4 * L, 4 * L),) * 3, n_sets, 2), "fp32")
                off = torch.arange(n_sets + 1, dtype=torch.int64, device="cuda")
                nb = _lib.ap_adjoint_workspace_bytes(h.h, n_sets, 1, 1)
                ws = torch.empty((nb + 255) // 256 * 64, dtype=torch.float32, device="cuda")
                dJ = torch.zeros((n_sets, _lib.AP_NPARAM), dtype=torch.float64, device="cuda")
                J = torch.zeros(n_sets, dtype=torch.float64, device="cuda")
                stream.synchronize()
                start.wait()
                for _ in range(400):
                    _lib.ap_push_adjoint(h.h, parts, off, None, 0.0, 0.01, 1, 1, "fp32", dJ, J, ws, stream)
                stream.synchronize()
        except Exception as e:  # reported by the main thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(n,)) for n in (1, 4096)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
