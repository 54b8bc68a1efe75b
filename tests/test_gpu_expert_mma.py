"""GPU parity of the multi-token expert factors (mma.sync tiles of 8 and 16 tokens) at the sizes where
their tiling can go wrong: expert loads around a token group (1, 7, 8, 9, 15 .. 17, 33), one and several
row blocks and runs of row blocks, several segments, K-step remainders of every bit-width, odd expert
counts, all scale groups, and both sides of the decode batch and of the 256 tokens past which the down
kernel takes longer runs of row blocks.  Also the largest routing, waits that run out, and a routing
that is not the call's.

Tolerance: the operands are fp16 pairs (at least 21 bits) and the codes exact, so what remains is fp32
summation over at most n + I terms and the output basis' bf16 pair (2^-17 of each term of s): below
2^-17 sqrt(n) max|Phi s| / max|y| <= 1e-4 at these sizes.
"""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu
TOL = 1e-4
BITS = {0: 0.1, 1: 0.15, 2: 0.2, 3: 0.15, 4: 0.15, 6: 0.15, 8: 0.1}


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2606_00079_gb300 as bm
    torch.cuda.set_device(0)
    return torch, bm


@pytest.mark.parametrize("T,E,k,D,n,I,group,bits", [
    (3, 9, 2, 300, 260, 256, 128, BITS),        # three tokens, features not a multiple of 8
    (3, 4, 3, 256, 200, 384, 64, BITS),
    (3, 8, 2, 128, 64, 128, 64, BITS),          # the smallest layer whose three and four tokens take the chain
    (4, 8, 2, 128, 64, 128, 64, BITS),
    (5, 33, 3, 96, 75, 128, 128, BITS),         # decode batch, one row block, odd expert count
    (8, 4, 2, 128, 200, 1152, 128, BITS),       # nine row blocks: a full and a partial run of the down kernel
    (8, 5, 1, 72, 61, 64, 32, BITS),            # rows past the units' length, four groups a row block
    (9, 33, 1, 64, 75, 384, 128, BITS),         # first size past the decode batch
    (17, 33, 2, 100, 90, 256, 64, BITS),        # odd expert count, tiles of 16, two groups a row block
    (33, 3, 1, 64, 130, 512, 256, BITS),        # groups of two row blocks
    (34, 2, 2, 256, 1100, 256, 128, {1: 1.0}),  # several segments of one bit-width
    (34, 2, 2, 64, 1030, 128, 128, {3: .5, 4: .5}),
    (40, 2, 1, 64, 515, 256, 32, {6: .5, 8: .5}),
    (257, 5, 2, 64, 75, 768, 128, BITS),        # past 256 tokens: one run of six row blocks, a ring of two stages
    (257, 3, 2, 64, 75, 1152, 128, BITS),       # runs of five and four row blocks
    (257, 3, 2, 64, 75, 1280, 256, BITS),       # runs of six and four, groups of two row blocks
    (300, 3, 2, 64, 75, 768, 32, BITS),         # runs of four and two, four groups a row block
])
def test_expert_tiles(env, T, E, k, D, n, I, group, bits):
    torch, bm = env
    spec = synth.scaled_spec(synth.WORKLOADS["tiny"], D=D, E=E, I=I, n=n, group=group, top_k=k)
    layer = (synth.make_layer(spec, seed=T + n, bits_dist=bits, alpha_scale=4.0) if n <= D
             else wide_layer(spec, T + n, bits))
    L = bm.bitsmoe_pack(layer, device=0)
    plan = bm.bitsmoe_forward_plan(L, T, k)
    assert plan == (bm.PLAN_DECODE_CHAIN | bm.PLAN_TC_PROJECTIONS if T <= 8 else
                    bm.PLAN_TC_PROJECTIONS | bm.PLAN_TC_GATE_UP | bm.PLAN_TC_DOWN)
    # The plan of the decode batch does not name its expert kernels.  They are these whenever 16 tokens take them:
    # the same layer and tiles of 8 tokens, and a shared-memory plan that grows with the routed experts alone.
    assert bm.bitsmoe_forward_plan(L, max(T, 16), k) & bm.PLAN_TC_GATE_UP
    x, logits = synth.make_inputs(spec, T, seed=T)
    # uneven loads: the first experts hold 1, 7, 8, 9, .. of the first choices
    e, t = 0, 0
    for load in (1, 7, 8, 9, 15, 17, 33):
        logits[t:t + load, e % E] += 10.0
        e, t = e + 1, t + load
    ws = bm.Workspace(L, T, k)
    for _ in range(2):   # the second call on a used workspace
        y = bm.moe_forward(L, torch.from_numpy(x.view(np.int16)).cuda(), torch.from_numpy(logits).cuda(), k, ws=ws)
    torch.cuda.synchronize()
    assert bm.bitsmoe_last_device_status(ws.ptr) == 0
    ref = oracle.moe_forward_factored(layer, x, logits, k)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("E", [1, 3])
def test_most_pairs(env, E):
    """The router takes P + 2 E < 51200 pairs (its places inside an expert's list have 16 bits): the last accepted
    call, with nearly all tokens on one expert, against the oracle; one pair more, and past 65536, is refused."""
    torch, bm = env
    spec = synth.scaled_spec(synth.WORKLOADS["tiny"], D=64, E=E, I=64, n=48, group=64, top_k=1)
    layer = synth.make_layer(spec, seed=E, bits_dist=BITS, alpha_scale=4.0)
    L = bm.bitsmoe_pack(layer, device=0)
    T = 51200 - 2 * E - 1
    x, logits = synth.make_inputs(spec, T, seed=E)
    logits[:, 0] += 100.0
    logits[7::1000, E - 1] += 200.0
    y = bm.moe_forward(L, torch.from_numpy(x.view(np.int16)).cuda(), torch.from_numpy(logits).cuda(), 1)
    ref = oracle.moe_forward_factored(layer, x, logits, 1)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= TOL * np.max(np.abs(ref))
    for over in (T + 1, 70000):
        x2 = torch.zeros((over, spec.D), dtype=torch.int16, device="cuda")
        lg = torch.zeros((over, E), dtype=torch.float32, device="cuda")
        with pytest.raises(bm.BitsMoEError) as err:
            bm.moe_forward(L, x2, lg, 1)
        assert err.value.code == bm.ERR_CODE["SHAPE"]


@pytest.mark.parametrize("T,E,k,n,I", [(16, 8, 8, 1100, 1152), (600, 2, 2, 1100, 256)])   # tiles of 8 and of 16 tokens
def test_waits_that_run_out(env, T, E, k, n, I):
    """Block 0 of both expert kernels leaves out the arrivals at its first stage (testing hook) and every wait inside
    a block is bounded to about a millisecond: both kernels return after it (their copies in flight waited for), the
    status word reports TIMEOUT, and the next call on the same workspace is correct."""
    torch, bm = env
    spec = synth.scaled_spec(synth.WORKLOADS["tiny"], D=64, E=E, I=I, n=n, group=128, top_k=k)
    layer = wide_layer(spec, T, {4: 1.0})
    L = bm.bitsmoe_pack(layer, device=0)
    assert bm.bitsmoe_forward_plan(L, T, k) & bm.PLAN_TC_GATE_UP
    x, logits = synth.make_inputs(spec, T, seed=T)
    xd, ld = torch.from_numpy(x.view(np.int16)).cuda(), torch.from_numpy(logits).cuda()
    ws = bm.Workspace(L, T, k)
    y = torch.empty((T, spec.D), dtype=torch.float32, device="cuda")
    clocks = 2_000_000
    bm.bitsmoe_debug_wait_limit(1, clocks)
    try:
        ms = bm.bitsmoe_profile_forward(xd.data_ptr(), ld.data_ptr(), T, k, L, y.data_ptr(), ws.ptr, ws.nbytes,
                                        torch.cuda.current_stream().cuda_stream)
    finally:
        bm.bitsmoe_debug_wait_limit(0, 0)
    assert 0.4 * clocks / 1e6 < min(ms[2:4]) and max(ms[2:4]) < 500, ms   # gate/up and down (SM clock up to 2.1 GHz)
    assert bm.bitsmoe_last_device_status(ws.ptr) == bm.ERR_CODE["TIMEOUT"]
    y = bm.moe_forward(L, xd, ld, k, ws=ws)
    assert bm.bitsmoe_last_device_status(ws.ptr) == 0
    ref = oracle.moe_forward_factored(layer, x, logits, k)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("D", [4096, 4098])   # tokens copied by TMA, and staged by warps
def test_projection_waits_that_run_out(env, D):
    """The first CTA of the tensor-core projection never reports its first ring slot free (testing hook): the kernel
    returns within the bounds of its waits, the status word reports TIMEOUT, and the next call is correct."""
    torch, bm = env
    T = 256
    spec = synth.scaled_spec(synth.WORKLOADS["tiny"], D=D, E=2, I=64, n=64, group=64, top_k=1)
    layer = synth.make_layer(spec, seed=D, bits_dist=BITS, alpha_scale=4.0, basis_method="householder")
    L = bm.bitsmoe_pack(layer, device=0)
    x, logits = synth.make_inputs(spec, T, seed=D)
    xd, ld = torch.from_numpy(x.view(np.int16)).cuda(), torch.from_numpy(logits).cuda()
    ws = bm.Workspace(L, T, 1)
    y = torch.empty((T, D), dtype=torch.float32, device="cuda")
    clocks = 2_000_000
    bm.bitsmoe_debug_wait_limit(1, clocks)
    try:
        ms = bm.bitsmoe_profile_forward(xd.data_ptr(), ld.data_ptr(), T, 1, L, y.data_ptr(), ws.ptr, ws.nbytes,
                                        torch.cuda.current_stream().cuda_stream)
    finally:
        bm.bitsmoe_debug_wait_limit(0, 0)
    assert 0.4 * clocks / 1e6 < ms[1] < 500, ms
    assert bm.bitsmoe_last_device_status(ws.ptr) == bm.ERR_CODE["TIMEOUT"]
    y = bm.moe_forward(L, xd, ld, 1, ws=ws)
    assert bm.bitsmoe_last_device_status(ws.ptr) == 0
    ref = oracle.moe_forward_factored(layer, x, logits, 1)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("T", [8, 40])
def test_impossible_routing_is_refused(env, T):
    """A routing whose experts hold more tokens than the call has (testing hook) is left out and reported as
    WORKSPACE_STATE; the next call on the same workspace is correct."""
    torch, bm = env
    spec = synth.scaled_spec(synth.WORKLOADS["tiny"], D=128, E=8, I=256, n=96, group=128, top_k=3)
    layer = synth.make_layer(spec, seed=T, bits_dist=BITS, alpha_scale=4.0)
    L = bm.bitsmoe_pack(layer, device=0)
    x, logits = synth.make_inputs(spec, T, seed=T)
    xd, ld = torch.from_numpy(x.view(np.int16)).cuda(), torch.from_numpy(logits).cuda()
    ws = bm.Workspace(L, T, spec.top_k)
    bm.bitsmoe_debug_bounds(2)
    try:
        bm.moe_forward(L, xd, ld, spec.top_k, ws=ws)
        assert bm.bitsmoe_last_device_status(ws.ptr) == bm.ERR_CODE["WORKSPACE_STATE"]
    finally:
        bm.bitsmoe_debug_bounds(0)
    y = bm.moe_forward(L, xd, ld, spec.top_k, ws=ws)
    assert bm.bitsmoe_last_device_status(ws.ptr) == 0
    ref = oracle.moe_forward_factored(layer, x, logits, spec.top_k)
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= TOL * np.max(np.abs(ref))


@pytest.mark.parametrize("e", [-56, 57])
@pytest.mark.parametrize("T,E,k,D,n,I,group", [
    (4, 8, 2, 256, 256, 512, 64), (8, 16, 4, 256, 200, 384, 128), (40, 32, 8, 128, 100, 128, 32), (70, 8, 2, 512, 300, 256, 128)])
def test_tiny_and_huge_activations(env, T, E, k, D, n, I, group, e):
    """Tokens scaled by 2^e: h = SiLU(gate) * up near 2^-112 and 2^118, whose power-of-two scaling into fp16's range
    takes the largest exponents.  Tolerance: that of ordinary tokens, and for the tiny ones fp32 additions into global
    memory and bf16 products, which drop what lies below 2^-126: at most k + 1 such errors an element of s, uniform,
    through rows of Phi of norm at most 1: four standard deviations."""
    torch, bm = env
    spec = synth.scaled_spec(synth.WORKLOADS["tiny"], D=D, E=E, I=I, n=n, group=group, top_k=k)
    layer = synth.make_layer(spec, seed=3, bits_dist=BITS, alpha_scale=4.0)
    L = bm.bitsmoe_pack(layer, device=0)
    x, logits = synth.make_inputs(spec, T, seed=9)
    xf = (x.astype(np.uint32) << 16).view(np.float32) * np.float32(2.0) ** e
    x = synth.f32_to_bf16_bits(xf.astype(np.float32))
    y = bm.moe_forward(L, torch.from_numpy(x.view(np.int16)).cuda(), torch.from_numpy(logits).cuda(), k)
    with np.errstate(over="ignore"):   # exp of a huge gate in the oracle: SiLU is 0 there
        ref = oracle.moe_forward_factored(layer, x, logits, k)
    tol = TOL * np.max(np.abs(ref)) + 4.0 * np.sqrt((k + 1) / 3.0) * 2.0 ** -126
    assert np.max(np.abs(y.cpu().numpy() - ref)) <= tol


def wide_layer(spec, seed, bits):
    """A layer with more units than features (n > D): random bases of norm-1 columns."""
    layer = synth.make_layer(synth.scaled_spec(spec, D=spec.n), seed=seed, bits_dist=bits, alpha_scale=4.0,
                             basis_method="householder")
    rng = np.random.default_rng(seed)
    b = rng.standard_normal((3, spec.D, spec.n)) / np.sqrt(spec.D)
    layer.update(D=spec.D, basis=synth.f32_to_bf16_bits(b.astype(np.float32)))
    return layer
