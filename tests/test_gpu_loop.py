"""The decoding loop in one kernel (csrc/bv_loop.cu) at the edges of its sizes, against the loop of one launch a step (GPU)."""
import pytest
import torch

from paper_2403_10444_b200 import specdec, workloads as wl

pytestmark = pytest.mark.gpu


# rows of one vector; of fewer vectors than streaming warps; one beyond whole runs of 32 vectors a warp; uneven parts; the
# sampler's two forms (2048 vectors a row); positions beyond 32; the largest rows of which two fit in shared memory, and the
# next larger ones, which take the loop of two launches an iteration
@pytest.mark.parametrize("dtype,V,B,gamma,N", [("bf16", 8, 5, 1, 6), ("bf16", 40, 9, 3, 5), ("f32", 2052, 7, 5, 4), ("bf16", 4104, 33, 4, 4), ("bf16", 16376, 8, 2, 3),
                                               ("bf16", 16384, 150, 3, 3), ("f32", 8192, 6, 34, 2), ("bf16", 1024, 3, 64, 3), ("f32", 26624, 3, 2, 2), ("f32", 26628, 3, 2, 2)])
@pytest.mark.parametrize("sigma_d", [0.2, 1.0])
def test_one_kernel_generates_what_the_steps_generate(dtype, V, B, gamma, N, sigma_d):
    import paper_2403_10444_b200 as bv
    tt, dt = wl.markov_models(V, dtype, V + gamma, 2.0, sigma_d, 1.1 if V > 8 else 0.0, "cuda")
    ud, uv = wl.loop_uniforms(N, B, gamma, V, "cuda")
    first = torch.arange(B, dtype=torch.int32, device="cuda") % V
    for algo in specdec.ALGOS:
        a = specdec.run(tt, dt, first, ud, uv, gamma, 0.9, algo)
        assert bv.bv_last_launch_count() == (1 if V != 26628 else 2 * N + 1)
        b = specdec.run(tt, dt, first, ud, uv, gamma, 0.9, algo, chain=False)
        # (their sums run in another order: at most 1e-4 + 2e-8 V of the draws lie so close to the edge of a token's cell that
        # this moves them, and such a sequence goes its own way from there on)
        draws = N * B * (gamma + 1)
        same = sum(torch.equal(a["tokens"][s], b["tokens"][s]) for s in range(B))
        assert same >= B - 1 - int(draws * (1e-4 + 2e-8 * V)), (algo, same)
        for s in range(B):
            if torch.equal(a["tokens"][s], b["tokens"][s]):
                assert a["lengths"][s] == b["lengths"][s] and torch.equal(a["tau"][:, s], b["tau"][:, s]) and torch.equal(a["drafted"][:, s], b["drafted"][:, s])


@pytest.mark.parametrize("algo", specdec.ALGOS)
def test_rows_that_cannot_be_read(algo):
    # a NaN in the target row that a sequence's blocks start from: no iteration of any algorithm can use it
    V, B = 256, 6
    tt, dt = wl.markov_models(V, "f32", 3, 2.0, 0.7, 1.1, "cuda")
    ud, uv = wl.loop_uniforms(2, B, 3, 4, "cuda")
    first = torch.full((B,), 2, dtype=torch.int32, device="cuda")
    specdec.run(tt, dt, first, ud, uv, 3, algo=algo)
    bad = tt.clone()
    bad[2, 7] = float("nan")
    with pytest.raises(RuntimeError):
        specdec.run(bad, dt, first, ud, uv, 3, algo=algo)
