"""Device memory that only speeds calls up (the partials of short source
chunks, the operands of the tensor-core far field): taken where there is room,
given up without a trace where there is none or another allocation needs it."""
import numpy as np
import pytest

from synth import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    from paper_1910_01011_gb300 import api as a
    return a


def device_vectors(s, R):
    import torch
    return torch.from_numpy(np.stack([scenes.smooth_trace_vector(s, r) for r in range(R)])).cuda()


def error_text(c):
    return c.lib.bem_last_error(c.h)


def test_long_chunks_leave_the_rest_alone(api):
    """640 tiles: the partials of short source chunks take 0.74 GB, those of
    four chunks 55 MB.  Under a budget for the latter only, beside the operands
    of a product of two vectors: one-vector products have the bits of the long
    chunks, the second allocates nothing, the operands stay in place (same bits
    as without a budget), and no error text is left behind."""
    s = scenes.sphere_scene(5)
    X = device_vectors(s, 2)
    c = api.Context.from_scene(s)
    ref2 = c.apply(X, precision=api.FP32)
    used = c.memory()[0]
    c.close()
    c = api.Context.from_scene(s, chunk_tiles=160)
    ref1 = c.apply(X[0].contiguous(), precision=api.FP32)
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used + (100 << 20))
    assert (c.apply(X, precision=api.FP32) == ref2).all()
    assert (c.apply(X[0].contiguous(), precision=api.FP32) == ref1).all()
    held = c.memory()
    assert (c.apply(X[0].contiguous(), precision=api.FP32) == ref1).all()
    assert c.memory() == held
    assert (c.apply(X, precision=api.FP32) == ref2).all()
    assert error_text(c) == b""
    c.close()


def test_short_chunks_make_room(api):
    """Partials of short source chunks that fit at first go when a later call
    needs the room, and the product after it takes the long chunks."""
    s = scenes.sphere_scene(5)
    x = device_vectors(s, 1)[0]
    c = api.Context.from_scene(s)
    short = c.apply(x, precision=api.FP32)
    used = c.memory()[0]
    c.close()
    c = api.Context.from_scene(s, chunk_tiles=160)
    long = c.apply(x, precision=api.FP32)
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used + (1 << 20))
    assert (c.apply(x, precision=api.FP32) == short).all()
    c.apply(x, precision=api.FP64)  # split vectors beside the partials
    c.apply(x, op=api.PREC)         # vectors of the sparse solves
    y = c.apply(x, precision=api.FP32)
    assert (y == short).all() or (y == long).all()
    assert c.memory()[1] <= used + (1 << 20)
    c.close()


def test_tensor_core_operands_come_back(api):
    """The operands of several vectors' products go when another allocation
    needs their room (vectors staged from the host), and are there again, with
    the same bits, once that room is free."""
    s = scenes.sphere_scene(4)
    X = device_vectors(s, 16)
    c = api.Context.from_scene(s)
    ref = c.apply(X, precision=api.FP32)
    used = c.memory()[0]
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used + (1 << 20))
    assert (c.apply(X, precision=api.FP32) == ref).all()
    y = c.apply(X.cpu().numpy(), precision=api.FP32)  # 2.6 MB of staging
    assert np.linalg.norm(y - ref.cpu().numpy()) < 1e-5 * np.linalg.norm(y)
    assert c.memory()[0] < used - (1 << 22)
    assert (c.apply(X, precision=api.FP32) == ref).all()
    assert error_text(c) == b""
    c.close()


def test_no_room_for_the_operands(api):
    """A budget that misses the operands of 16 vectors by 4 MiB: the product by
    the FP32 kernel alone, nothing of the tensor cores' memory held, no error
    text, and nothing allocated by the second product."""
    s = scenes.sphere_scene(4)
    X = device_vectors(s, 16)
    c = api.Context.from_scene(s)
    ref = c.apply(X, precision=api.FP32)
    used = c.memory()[0]
    c.close()
    c = api.Context.from_scene(s, hbm_budget_bytes=used - (1 << 22))
    y = c.apply(X, precision=api.FP32)
    assert (y - ref).norm() < 1e-5 * ref.norm()
    assert error_text(c) == b""
    held = c.memory()
    assert (c.apply(X, precision=api.FP32) == y).all()
    assert c.memory() == held
    assert error_text(c) == b""
    c.close()


def test_estimate_counts_what_a_solve_needs(api):
    """640 tiles: the solve's estimate is that of the longest source chunks,
    and the solve runs under it."""
    s = scenes.sphere_scene(5)
    kw = dict(precision=api.FP32, tol=1e-3, operator_mode=0, max_iter=60)
    est = []
    for chunk in (160, 0):
        c = api.Context.from_scene(s, chunk_tiles=chunk, r_eps=0.2)
        est.append(c.estimate_solve_bytes(1, **kw))
        c.close()
    assert est[0] == est[1]
    c = api.Context.from_scene(s, hbm_budget_bytes=est[0], r_eps=0.2)
    c.set_plane_wave((0, 0, 1))
    c.solve(**kw)
    assert c.memory()[1] <= est[0]
    c.close()


@pytest.mark.parametrize("share", [1.25, 3.5])
def test_served_scenes_share_a_budget(api, share):
    """Two scenes whose matrix-free solves of eight excitations take the
    tensor-core far field where the budget has room, under one that holds a
    little more than one of them (idle scenes are evicted) and one that holds
    both running: every request completes, within the budget, with the
    solutions found without a limit."""
    tr = scenes.bowl_transducer(seed=0, n_elem=6, R=4.0, aperture=3.0, piston_radius=0.3, gap=0.05)
    kw = dict(precision=api.FP32, tol=1e-8, operator_mode=0, batch_rhs=8, block_gmres=1)
    W = [np.exp(2j * np.pi * np.random.default_rng(i).random((8, 6))) for i in range(2)]

    def serve(budget, rounds):
        srv = api.Server(slots=2, max_batch_rhs=8, hbm_budget_bytes=budget, join=0, **kw)
        ids = [srv.add_scene(scenes.sphere_scene(4, k0=4.0 + i), transducer=tr, omega_rho0=2.6, r_eps=0.2) for i in range(2)]
        est = max(srv.estimate(i, 8) for i in ids)
        hs = [(i, srv.submit(ids[i], W[i])) for _ in range(rounds) for i in range(2)]
        out = {}
        for i, h in hs:
            assert srv.wait(h, 600) == 2, srv.error(h)
            out[i] = srv.result(h, 8, ids[i])[0]
        st = srv.stats()
        srv.close()
        assert st["completed"] == 2 * rounds and st["failed"] == 0
        assert budget == 0 or st["peak_device_bytes"] <= budget
        return out, est

    ref, est = serve(0, 1)
    out, _ = serve(int(share * est), 3)
    for i in range(2):
        assert np.linalg.norm(out[i] - ref[i]) < 1e-6 * np.linalg.norm(ref[i])
