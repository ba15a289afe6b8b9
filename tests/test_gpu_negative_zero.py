"""Settings of -0.0 are settings of 0: validation accepts them (they are not below 0), so the solve
and the evaluation give bitwise what 0.0 gives, in every form."""
import numpy as np
import pytest

from paper_2606_31098_gb300 import binding as B
from paper_2606_31098_gb300 import scenes as S

from gpu_support import device_frame, require_cuda

pytestmark = pytest.mark.gpu

FIELDS = ("min_valid_frac", "gate_grav", "gate_range")


@pytest.fixture(scope="module")
def torch():
    return require_cuda()


def frame(side, n_hyps=5):
    """A frame whose gravity reading is off, so that a gate would close."""
    f = S.make_frame(S.config_reduced_frame(crop_side=side, n_hyps=n_hyps), S.frame_seed(2, 970))
    g = f.gravity_cam + np.array([0.0, 0.08, 0.0])
    return f.replace(gravity_cam=g / np.linalg.norm(g))


def options(zero, names):
    kw = dict(min_valid_frac=0.0, gate_grav=0.0, gate_range=0.0)
    kw.update({k: zero for k in names})
    return B.Options(iters=(3, 3, 2), max_points=12000, max_hyps=10, max_frames=2, **kw)


def outputs(torch, opts, fa, two):
    s = B.Solver(opts)
    res = [s.solve(fa), s.solve(two), s.solve_batch([fa])[0], *s.solve_batch([fa, two])]
    out = [np.concatenate([r.T_cw.ravel(), r.cost, r.n_valid, r.status, [r.best]]) for r in res]
    T = np.ascontiguousarray(fa.arrays["T_cw"].cpu().numpy())
    out.append(s.normal_eq(fa, 0, T))
    ne = torch.zeros((fa.M, 29), dtype=torch.float64, device="cuda")
    B.check(B.normal_eq_noalloc(opts, fa, 0, fa.arrays["T_cw"], ne))
    out.append(ne.cpu().numpy())
    s.close()
    server = B.Server(opts, 1 << 30, 2)
    r = server.wait(server.submit(fa))[0]
    out.append(np.concatenate([r.T_cw.ravel(), r.cost, r.n_valid, r.status, [r.best]]))
    server.close()
    return out


@pytest.mark.parametrize("names", [FIELDS, *((n,) for n in FIELDS)], ids=lambda n: "+".join(n))
def test_negative_zero_is_zero(torch, names):
    """24^2 anchors: a level in one launch, a batch of one tile; 104^2: a launch per iteration, a
    batch of several tiles."""
    fa, two = device_frame(frame(24)), device_frame(frame(104))
    want, got = outputs(torch, options(0.0, names), fa, two), outputs(torch, options(-0.0, names), fa, two)
    for a, b in zip(want, got):
        np.testing.assert_array_equal(a, b)
    # the solves moved: a threshold that rejects every step would leave the starting poses
    assert not np.array_equal(want[0][:60], fa.arrays["T_cw"].cpu().numpy().ravel())
