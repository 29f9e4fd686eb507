"""A context's scratch starts every call as that call needs it, whatever the calls before left there:
two calls that overlap on one context (which no caller may let them) leave cell counts that are not
zero, and a later call in order has to give what a fresh context gives, bit by bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2401_10462_gb300 import api
    return torch, api


def _call(env, ctx, kind, sizes, gen):
    torch, api = env
    mols = [gen.make("globule", n, 3 + n % 5) for n in sizes]
    x = torch.as_tensor(np.concatenate([m.coords for m in mols]), device="cuda")
    r = torch.as_tensor(np.concatenate([m.radii for m in mols]), device="cuda")
    a, g = torch.empty_like(r), torch.empty_like(x)
    if kind == "sr":
        ctx.compute_sr(x, r, torch.as_tensor(gen.sphere_points(96), device="cuda"), a)
        g.zero_()
    elif kind == "batch":
        ctx.compute_batch(np.cumsum([0] + list(sizes)), x, r, a, g)
    else:
        ctx.compute(x, r, a, g)
    ctx.status_sync()
    return a.cpu().numpy(), g.cpu().numpy()


@pytest.mark.parametrize("kind,sizes,options", [
    ("one", (300,), {}), ("one", (2049,), {}), ("one", (17001,), {}), ("sr", (2500,), {}),
    ("one", (5003,), {"skin": 1.0}), ("one", (3001,), {"max_cells": 20000}), ("one", (2500,), {"max_atoms": 20000}),
    ("batch", (300, 2500, 1, 40), {}), ("batch", (17, 5000), {"skin": 0.5})])
def test_counts_left_over(env, gen, kind, sizes, options):
    _, api = env
    ctx, fresh = api.Context(**options), api.Context(**options)
    _call(env, ctx, kind, sizes, gen)                        # allocates
    ctx._raise(api._lib.dsasa_debug_disturb_counts(ctx._h))
    if "skin" in options:                                    # another probe: the lists are not reused
        _call(env, ctx, "sr", (12,), gen)
    got = _call(env, ctx, kind, sizes, gen)
    again = _call(env, ctx, kind, sizes, gen)
    ref = _call(env, fresh, kind, sizes, gen)
    ctx.close()
    fresh.close()
    assert np.array_equal(got[0], ref[0]) and np.array_equal(got[1], ref[1])
    if "skin" not in options:
        assert np.array_equal(again[0], ref[0]) and np.array_equal(again[1], ref[1])
