"""Several RK3 steps in one call, and states on addresses that are only 8-byte aligned: the
branches of the FP32 operator that one step on an aligned state does not reach."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_2207_11571_gb300 import inputs  # noqa: E402


@pytest.fixture(scope="module")
def dg():
    from tests.libbuild import ensure_built
    ensure_built()
    from paper_2207_11571_gb300 import dg as _dg
    _dg.lib()
    return _dg


def state(dg, ctx, N):
    q = torch.empty(5 * N, dtype=torch.float64, device="cuda")
    dg.dg_init_tgv(ctx, q, torch.from_numpy(inputs.perturbation((5, N), eps=1e-3).ravel()).cuda())
    return q


@pytest.mark.parametrize("K,P,les,split,prec", [(4, 3, 0, 0, 1), (3, 3, 1, 0, 1), (3, 3, 0, 1, 1), (5, 1, 0, 0, 1),
                                                (3, 2, 1, 0, 1), (3, 4, 0, 0, 1), (2, 5, 1, 0, 1), (3, 6, 0, 0, 1),
                                                (2, 7, 0, 0, 1), (2, 8, 0, 1, 1), (3, 3, 0, 0, 0)])
def test_steps_in_one_call_equal_single_steps(dg, K, P, les, split, prec):
    """Within a call the FP32 operator's last stage also forms the next step's stage state
    (in the other buffer); the same conversions, so the same bits as a step per call."""
    N = K ** 3 * (P + 1) ** 3
    ctx = dg.dg_create(K, P, 400.0, 0.1, 0.71, les, precision=prec, volume_flux=split)
    try:
        q = state(dg, ctx, N)
        dt = dg.dg_stable_dt(ctx, q, 0.5)
        one, many = q.clone(), q.clone()
        for _ in range(5):
            dg.dg_rk3_step(ctx, one, dt, 1)
        dg.dg_rk3_step(ctx, many, dt, 3)   # an odd number of steps leaves the buffers exchanged
        dg.dg_rk3_step(ctx, many, dt, 2)
        torch.cuda.synchronize()
        assert torch.isfinite(many).all() and not torch.equal(many, q)
        assert torch.equal(many, one)
    finally:
        dg.dg_destroy(ctx)


@pytest.mark.parametrize("K", [3, 4])
def test_state_on_an_8_byte_boundary_equals_an_aligned_one(dg, K):
    """At P = 3 the FP64 state moves in 16-byte vectors where its address allows."""
    P, N = 3, K ** 3 * 64
    ctx = dg.dg_create(K, P, 400.0, 0.1, 0.71, 0, precision=1)
    try:
        q = state(dg, ctx, N)
        buf = torch.empty(5 * N + 1, dtype=torch.float64, device="cuda")
        odd = buf[1:]
        odd.copy_(q)
        R, Rbuf = torch.empty_like(q), torch.empty(5 * N + 1, dtype=torch.float64, device="cuda")
        dg.dg_rhs(ctx, q, R)
        dg.dg_rhs(ctx, odd, Rbuf[1:])
        dg.dg_rk3_step(ctx, q, 1e-3, 2)
        dg.dg_rk3_step(ctx, odd, 1e-3, 2)
        torch.cuda.synchronize()
        assert torch.equal(Rbuf[1:], R) and torch.equal(odd, q)
    finally:
        dg.dg_destroy(ctx)


@pytest.mark.parametrize("K,P,prec", [(3, 3, 1), (11, 3, 1), (12, 3, 1), (14, 3, 1), (15, 3, 1), (16, 3, 1), (17, 3, 1),
                                      (13, 3, 0), (14, 3, 0), (11, 2, 0), (14, 2, 0)])
def test_phase_b_blocks_of_every_size_give_the_same_bits(dg, K, P, prec):
    """Phase B takes 2, 4 or 8 elements per block (FP64 also cubes) by the size of the mesh;
    a batch always takes the widest rows.  Each face term is the same arithmetic."""
    b = dg.dg_create_batch([(K, P, 400.0, 0.1, 0.71, 0), (3, P, 200.0, 0.1, 0.71, 0)], precision=prec)
    try:
        qs = [state(dg, dg.dg_batch_member(b, i), k ** 3 * (P + 1) ** 3) for i, k in enumerate((K, 3))]
        alone = qs[0].clone()
        dt = 1e-3
        dg.dg_batch_rk3_step(b, qs, [dt, dt], 2)
        dg.dg_rk3_step(dg.dg_batch_member(b, 0), alone, dt, 2)
        torch.cuda.synchronize()
        assert torch.isfinite(alone).all()
        if prec == 1:
            assert torch.equal(alone, qs[0])
        else:   # separate compilations may contract a multiply-add differently: a rounding of the state
            assert (alone - qs[0]).abs().max().item() <= 4e-16 * alone.abs().max().item()
    finally:
        dg.dg_batch_destroy(b)


@pytest.mark.parametrize("K,P,first,nv,split", [(6, 3, 0, 5, 0), (5, 3, 1, 3, 0), (5, 3, 0, 5, 1), (6, 2, 0, 5, 0),
                                                (4, 5, 1, 3, 0)])
def test_corrected_steps_in_one_call_equal_single_steps_and_one_rhs(dg, K, P, first, nv, split):
    """The network runs ahead of phase A where the stage state and its features exist: within a
    call phase B writes both, at the start of a call the state pass (P = 3) or phase A does.
    The same features, so the same bits; and the forced dq/dt of a call on its own agrees
    with the per-layer path, which forms the features from the state after phase A."""
    from paper_2207_11571_gb300 import nn
    N, feat = K ** 3 * (P + 1) ** 3, nv * (P + 1) ** 3
    dims = [feat, 64, 64, feat]
    ctx = dg.dg_create(K, P, 400.0, 0.1, 0.71, 0, precision=1, volume_flux=split)
    net = nn.nn_create(feat, feat, 64, 2, first, nv, K ** 3, inputs.uniform_draws(dims, 3))
    try:
        # a forcing of order 0.1: larger ones drive the density negative within the steps
        nn.nn_set_scalers(net, *[v * torch.ones(feat).numpy() for v in (0.0, 1.0, 0.0, 1e-3)])
        q = state(dg, ctx, N)
        dt = dg.dg_stable_dt(ctx, q, 0.5)
        single, many, free = q.clone(), q.clone(), q.clone()
        for _ in range(3):
            dg.dg_rk3_step(ctx, single, dt, 1, net)
        dg.dg_rk3_step(ctx, many, dt, 3, net)
        dg.dg_rk3_step(ctx, free, dt, 3)
        torch.cuda.synchronize()
        assert torch.isfinite(many).all() and not torch.equal(many, free)
        assert torch.equal(many, single)
        R, Rl = torch.empty_like(q), torch.empty_like(q)
        dg.dg_rhs(ctx, q, R, net)
        nn.nn_set_fused(net, 0)   # a GEMM per layer
        dg.dg_rhs(ctx, q, Rl, net)
        plain = torch.empty_like(q)
        dg.dg_rhs(ctx, q, plain)
        torch.cuda.synchronize()
        # both paths sum the same bf16 products in FP32: the forcing itself to 1e-5, on top of
        # FP32 rounding of dq/dt
        forcing = (R - plain).abs().max().item()
        assert forcing > 0
        assert (R - Rl).abs().max().item() <= 1e-3 * forcing + 1e-6 * plain.abs().max().item()
    finally:
        nn.nn_destroy(net)
        dg.dg_destroy(ctx)


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("sides", ["both", "one"])
def test_negative_density_gives_nan(dg, prec, sides):
    """A flow that has left the physical states is told by NaN, also where the densities (and
    pressures) on both sides of a face are negative and their product is not."""
    K, P = 3, 3
    N = K ** 3 * (P + 1) ** 3
    ctx = dg.dg_create(K, P, 400.0, 0.1, 0.71, 0, precision=prec)
    try:
        q = state(dg, ctx, N)
        if sides == "both":
            q.neg_()
        else:
            q.view(5, K ** 3, -1)[:, 13].neg_()
        R = torch.empty_like(q)
        dg.dg_rhs(ctx, q, R)
        faces = R.view(5, K ** 3, 4, 4, 4)[:, 13, 0]
        torch.cuda.synchronize()
        assert torch.isnan(faces).all()
    finally:
        dg.dg_destroy(ctx)


def test_current_stream_handle_follows_torch_and_costs_little(dg):
    """At 8^3/P3 and below a call is bound by the host: the state pass added a launch to it, and
    looking the current stream up as an object costs more than that launch."""
    import time
    st = torch.cuda.Stream()
    assert not dg.stream_ptr().value == st.cuda_stream
    with torch.cuda.stream(st):
        assert dg.stream_ptr().value == st.cuda_stream == torch.cuda.current_stream().cuda_stream
        assert dg.stream_ptr(torch.cuda.default_stream()).value in (None, 0)
    assert dg.stream_ptr().value in (None, 0)

    def us(f, n=2000):
        best = float("inf")
        for _ in range(5):
            t = time.perf_counter()
            for _ in range(n):
                f()
            best = min(best, time.perf_counter() - t)
        return best / n * 1e6

    assert us(dg.stream_ptr) < 0.8 * us(torch.cuda.current_stream)


@pytest.mark.parametrize("K,P,prec", [(3, 3, 1), (12, 3, 1), (15, 3, 1), (2, 6, 1), (5, 6, 1), (3, 7, 1), (5, 7, 1), (1, 8, 1),
                                      (5, 8, 1), (5, 6, 0), (3, 7, 0), (5, 8, 0)])
def test_phase_b_blocks_of_a_mesh_and_of_a_large_batch_give_the_same_bits(dg, K, P, prec):
    """A batch takes its blocks by the elements of all members: beside a large one the widest
    (P = 3) or those of many elements per SM (P >= 6), where the mesh alone takes small blocks or
    a thread per node.  Each face term is the same arithmetic."""
    other = 20 if P == 3 else 6
    b = dg.dg_create_batch([(K, P, 400.0, 0.1, 0.71, 0), (other, P, 200.0, 0.1, 0.71, 0)], precision=prec)
    try:
        qs = [state(dg, dg.dg_batch_member(b, i), k ** 3 * (P + 1) ** 3) for i, k in enumerate((K, other))]
        alone = qs[0].clone()
        dg.dg_batch_rk3_step(b, qs, [1e-3, 1e-3], 2)
        dg.dg_rk3_step(dg.dg_batch_member(b, 0), alone, 1e-3, 2)
        torch.cuda.synchronize()
        assert torch.isfinite(alone).all()
        if prec == 1:
            assert torch.equal(alone, qs[0])
        else:   # separate compilations may contract a multiply-add differently: a rounding of the state
            assert (alone - qs[0]).abs().max().item() <= 4e-16 * alone.abs().max().item()
    finally:
        dg.dg_batch_destroy(b)


@pytest.mark.parametrize("P,prec", [(8, 0), (8, 1), (6, 0), (7, 0)])
def test_meshes_of_one_element_per_sm_take_the_same_time(dg, P, prec):
    """4^3 and 5^3 elements at P >= 6 are one block per SM in both phases, so they take the same
    time.  Interface blocks of a few warps took 1.2 to 1.3 times as long on 5^3; 1.12 leaves room
    for the larger launch."""
    def us(K):
        N = K ** 3 * (P + 1) ** 3
        ctx = dg.dg_create(K, P, 400.0, 0.1, 0.71, 0, precision=prec)
        try:
            q = state(dg, ctx, N)
            best = float("inf")
            for _ in range(6):
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record()
                for _ in range(30):
                    dg.dg_rk3_step(ctx, q, 1e-6)
                b.record()
                b.synchronize()
                best = min(best, a.elapsed_time(b) / 30 * 1e3)
            return best
        finally:
            dg.dg_destroy(ctx)
    small, large = us(4), us(5)
    assert large <= 1.12 * small, (small, large)


@pytest.mark.parametrize("K,split,width,hidden", [(16, 0, 512, 4), (13, 0, 256, 3), (10, 1, 256, 4), (6, 0, 128, 2)])
def test_phase_a_beside_the_network_equals_phase_a_before_it(dg, K, split, width, hidden):
    """Phase A reads the stage state while the network runs.  A network whose max_batch takes the
    elements in two parts goes after phase A, which then waits as usual; its clusters are the
    same, so every bit must be.  Many steps on changing states: a stale line is a wrong state."""
    from paper_2207_11571_gb300 import nn
    N, feat = K ** 3 * 64, 320
    dims = [feat] + [width] * hidden + [feat]
    ctx = dg.dg_create(K, 3, 400.0, 0.1, 0.71, 1, precision=1, volume_flux=split)
    draws = inputs.uniform_draws(dims, 5)
    nets = [nn.nn_create(feat, feat, width, hidden, 0, 5, rows, draws) for rows in (K ** 3, (K ** 3 + 1) // 2)]
    try:
        for net in nets:
            nn.nn_set_scalers(net, *[v * torch.ones(feat).numpy() for v in (0.0, 1.0, 0.0, 1e-4)])
        q = state(dg, ctx, N)
        dt = dg.dg_stable_dt(ctx, q, 0.4)
        beside, before, R, Rb = q.clone(), q.clone(), torch.empty_like(q), torch.empty_like(q)
        for steps in (1, 4, 2, 3, 1, 1, 5):
            dg.dg_rk3_step(ctx, beside, dt, steps, nets[0])
            dg.dg_rhs(ctx, beside, R, nets[0])
            dg.dg_rk3_step(ctx, before, dt, steps, nets[1])
            dg.dg_rhs(ctx, before, Rb, nets[1])
            torch.cuda.synchronize()
            assert torch.isfinite(before).all()
            assert torch.equal(beside, before) and torch.equal(R, Rb)
    finally:
        for net in nets:
            nn.nn_destroy(net)
        dg.dg_destroy(ctx)
