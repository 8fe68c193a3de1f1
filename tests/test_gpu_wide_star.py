"""A compartment with more children than 15 or 16 bits count: a star, the root
alone in its cell's top part and every child a subtree of its own."""
import numpy as np
import pytest

import oracle
from paper_1810_12742_gb300 import hines as H

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("children", [32767, 32768, 65535, 65536, 70000])
@pytest.mark.parametrize("mode", ["f64", "f32", "compensated", "packed f64", "cable solve"])
def test_every_child_is_counted(mode, children):
    import torch
    r = np.random.default_rng(81)
    n = children + 1
    p = np.zeros(n, np.int32)
    p[0] = -1
    a = r.uniform(0.5, 2.0, n)
    a[0] = 0.0
    s, g, b = r.uniform(0.01, 0.1, n), r.uniform(0.1, 1.0, n), r.uniform(-1, 1, n)
    s[0] = 0.1 * a.sum()
    d = s * (1.0 + 0.025 * g) + np.concatenate(([a.sum()], a[1:]))
    u = -a
    if mode in ("f32", "compensated"):
        d, u, b = (v.astype(np.float32).astype(np.float64) for v in (d, u, b))
    ref = oracle.solve_batch(np.array([n], np.int32), p, d, u, b)
    plan = H.Plan([n], p)
    t = torch.float32 if mode in ("f32", "compensated") else torch.float64
    dt, ut, bt, st, gt = (torch.as_tensor(v).cuda().to(t) for v in (d, u, b, s, g))
    if mode == "compensated":
        x = H.solve_compensated(plan, dt, ut, bt)
    elif mode == "packed f64":
        x = H.unpack(plan, H.solve_packed(plan, H.pack(plan, dt), H.pack_coupling(plan, ut), H.pack(plan, bt)))
    elif mode == "cable solve":
        x = H.cable_solve(plan, st, gt, ut, bt, 0.025, 1)
    else:
        x = H.solve(plan, dt, ut, bt)
    err = np.abs(x.cpu().numpy() - ref).max() / np.abs(ref).max()
    # one sum of `children` terms, one rounding each, over a pivot that keeps 1/50 of it, in front of the stated gates
    eps = np.finfo(np.float32 if mode == "f32" else np.float64).eps
    assert err <= max(50 * children * eps, {"f32": 1e-5, "compensated": 1e-10}.get(mode, 1e-12))
    assert plan.status() == 0
