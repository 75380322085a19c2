"""The FP64 push takes a coordinate's cell and CIC weight from integer arithmetic
where they cannot depend on the last bits of x / dx, and from the FP64
definition elsewhere.  Coordinates at the edges of that rule (nodes, ties of the
14-bit weight, their neighbouring doubles, the box's ends, tiny ones) for
several cell edges, gathered, pushed and deposited: bit for bit the oracle."""
import dataclasses

import numpy as np
import pytest

import oracle as O
import paper_1801_00972_gb300 as P
from paper_1801_00972_gb300 import build as B
from paper_1801_00972_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _edges(n, dx, top, rng, count):
    """count coordinates in [0, n dx), or [0, n dx] where top."""
    k = rng.integers(0, n, count)
    a = rng.integers(0, 16384, count)
    kind = np.arange(count) % 6
    base = np.select([kind == 0, kind == 1, kind == 2, kind == 3], [k * dx, (k + a / 16384.0) * dx, (k + (a + 0.5) / 16384.0) * dx,
                                                                    rng.random(count) * n * dx], rng.random(count) * 1e-9 * dx)
    step = rng.integers(-2, 3, count)
    x = np.where(step < 0, np.nextafter(base, -1.0), np.where(step > 0, np.nextafter(base, 1e9), base))
    x[:4] = [0.0, np.nextafter(n * dx, 0), 5e-324, n * dx if top else 0.0]
    hi = n * dx if top else np.nextafter(n * dx, 0)
    return np.clip(x, 0.0, hi)


@pytest.mark.parametrize("dx", [0.2e-3, 2.0 ** -12, 1.0 / 3000.0, 1.0000000000000002e-3, 7.7e-5])
def test_cells_and_weights_at_the_edges_match_the_oracle(dx):
    import torch
    B.build()
    torch.cuda.set_device(0)
    n = 6000
    wl = I.small(nx=8, ny=16, nz=32, n_e=n, n_i=n, grains=0, v_dc=-30.0, weight=1.0)
    wl = dataclasses.replace(wl, dx=dx)
    rng = np.random.default_rng(5)
    parts, base = [], 0
    for _ in range(2):
        x = np.stack([_edges(m, dx, a == 2, rng, n)[rng.permutation(n)] for a, m in enumerate((8, 16, 32))], 1)
        v = np.where(rng.random((n, 1)) < 0.5, 0.0, rng.standard_normal((n, 3)) * 0.1 * dx / wl.dt)
        parts.append((x, v, np.arange(base, base + n, dtype=np.uint32)))
        base += n
    ref = O.Sim(wl, parts)
    run = P.Run(wl, parts, prec=P.PIC_FP64, stream=torch.cuda.current_stream().cuda_stream)
    assert np.array_equal(run.rho(), ref.rho())
    phi = np.random.default_rng(6).standard_normal(wl.nodes)
    for s in (run, ref):
        s.set_phi(phi)
    for _ in range(2):
        run.advance()
        ref.advance()
        for sp in range(2):
            for a, b in zip(run.particles(sp), ref.particles(sp)):
                assert np.array_equal(a, b)
        assert np.array_equal(run.rho(), ref.rho())
    run.close()
