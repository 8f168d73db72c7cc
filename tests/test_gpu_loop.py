"""The decoding loop in one kernel (csrc/bv_loop.cu) at the edges of its sizes, against the loop of one launch a step (GPU)."""
import pytest
import torch

import oracle
from paper_2403_10444_b200 import specdec, workloads as wl
from parity import compare, run_oracle, to_numpy_logits

pytestmark = pytest.mark.gpu


def parts_at_a_near_tie(a, b, s, tt, dt, first, ud, uv, gamma, T, algo):
    """Where sequence s first differs between two runs of the loop: was that draw, or that test, within 1e-6 of its threshold?"""
    oalgo = oracle.TOKEN_VERIFY if algo.startswith("token") else oracle.BLOCK_VERIFY
    rows = lambda table, at: table[torch.as_tensor(at, device=table.device).long()].cpu()
    cur, pos = int(first[s]), 0
    for n in range(ud.shape[0]):
        da, db = a["drafted"][n, s].cpu(), b["drafted"][n, s].cpu()
        for i in range(gamma):
            if da[i] != db[i]:
                last = cur if i == 0 else int(da[i - 1])
                return oracle.sample_rows(to_numpy_logits(rows(dt, [last])), ud[n, i, s : s + 1].cpu().numpy(), T)[2][0] < 1e-6
        ta, tb = int(a["tau"][n, s]), int(b["tau"][n, s])
        ga, gb = a["tokens"][s, pos : pos + ta + 1].cpu(), b["tokens"][s, pos : pos + tb + 1].cpu()
        if ta != tb or not torch.equal(ga, gb):
            path = [cur] + da.tolist()
            inp = dict(target_logits=rows(tt, path)[None], draft_logits=rows(dt, path[:-1])[None], draft_tokens=da[None], uniforms=uv[n, s : s + 1].cpu(), temperature=T)
            ref = run_oracle(oalgo, inp)
            for tau, got in ((ta, ga), (tb, gb)):
                out = torch.full((1, gamma + 1), -1, dtype=torch.int32)
                out[0, : tau + 1] = got
                if compare(oalgo, ref, out, torch.tensor([tau + 1], dtype=torch.int32), None, inp).hard_mismatches:
                    return False
            return True
        cur, pos = int(ga[-1]), pos + ta + 1
    return False


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


# (the same calls, in one kernel whatever the shape says)
@pytest.mark.parametrize("dtype,V,B,gamma,N", [("bf16", 8, 5, 1, 6), ("bf16", 40, 9, 3, 5), ("f32", 2052, 7, 5, 4), ("bf16", 4104, 33, 4, 4), ("bf16", 16376, 8, 2, 3),
                                               ("bf16", 16384, 150, 3, 3), ("f32", 8192, 6, 34, 2), ("bf16", 1024, 3, 64, 3), ("f32", 26624, 3, 2, 2), ("f32", 26628, 3, 2, 2)])
@pytest.mark.parametrize("sigma_d", [0.2, 1.0])
def test_one_kernel_parts_from_the_steps_only_at_near_ties(dtype, V, B, gamma, N, sigma_d, bv_options):
    import paper_2403_10444_b200 as bv
    bv_options("loop", 1)
    T = 0.9
    tt, dt = wl.markov_models(V, dtype, V + gamma, 2.0, sigma_d, 1.1 if V > 8 else 0.0, "cuda")
    ud, uv = wl.loop_uniforms(N, B, gamma, V, "cuda")
    first = torch.arange(B, dtype=torch.int32, device="cuda") % V
    for algo in specdec.ALGOS:
        a = specdec.run(tt, dt, first, ud, uv, gamma, T, algo)
        assert bv.bv_last_launch_count() == (1 if V != 26628 else 2 * N + 1)
        b = specdec.run(tt, dt, first, ud, uv, gamma, T, algo, chain=False)
        # (their sums run in another order: at most 1e-4 + 2e-8 V of the draws lie so close to the edge of a token's cell that
        # this moves them, and such a sequence goes its own way from there on)
        same = lambda s: all(torch.equal(a[k][s] if k in ("tokens", "lengths") else a[k][:, s], b[k][s] if k in ("tokens", "lengths") else b[k][:, s]) for k in a)
        differ = [s for s in range(B) if not same(s)]
        assert len(differ) <= 1 + int(N * B * (gamma + 1) * (1e-4 + 2e-8 * V)), (algo, differ)
        for s in differ:
            assert parts_at_a_near_tie(a, b, s, tt, dt, first, ud, uv, gamma, T, algo), (algo, s)


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


# (32 sequences and fewer: whatever is selected, the last target row counts; more: where it is read)
@pytest.mark.parametrize("B,kernel", [(24, 4), (80, 5)])
@pytest.mark.parametrize("algo", range(4))
@pytest.mark.parametrize("gamma", [1, 4])
def test_faults_end_the_sequences_that_meet_them_and_no_others(B, kernel, algo, gamma, bv_options):
    # the draft goes from token t to t + 1, so that sequence b meets bad rows at position 40 - b and so on, or stops before it
    from paper_2403_10444_b200 import binding as bv
    V, N = 128, 2
    gen = torch.Generator().manual_seed(gamma)
    t = torch.randn((V, V), generator=gen)
    d = torch.full((V, V), -8.0)
    nxt = (torch.arange(V) + 1) % V
    t[torch.arange(V), nxt] += 4.0
    d[torch.arange(V), nxt] = 8.0
    t[40, 3], t[60, 5], d[50, 9], d[70] = float("nan"), float("inf"), float("nan"), float("-inf")
    tt, dt = t.cuda(), d.cuda()
    first = (36 + 2 * torch.arange(B) % 41).to(torch.int32)
    first[5], first[11] = V, -1
    ud, uv = wl.loop_uniforms(N, B, gamma, 7, "cuda")

    def run():
        return [x.cpu() for x in bv.bv_decode_loop(tt, dt, first.cuda(), ud, uv, gamma, 1.0, algo)]

    one = run()
    assert bv.bv_last_launch_count() == 1
    bv_options("kernel", kernel)
    two = run()
    assert bv.bv_last_launch_count() == 2 * N + 1 and bv.bv_last_kernel() == kernel
    for a, b in zip(one, two):
        assert torch.equal(a, b)
    tau = one[2]
    assert one[4][0] == 1 and (tau == -2).any() and (tau[0] >= 0).sum() >= B // 3
    if B > 32 and algo % 2 == 0:
        # the sequence that starts gamma before a target row that cannot be read is at fault only where that row is read
        last = [b for b in range(B) if first[b] + gamma in (40, 60)]
        assert last and all(tau[0, b] == -2 or tau[0, b] < gamma for b in last) and any(tau[0, b] >= 0 for b in last)


@pytest.mark.parametrize("algo", range(4))
def test_a_token_drawn_from_the_last_target_row_sees_every_vector(algo):
    # row 7 holds 2560 ones and, behind each of the first half of them, a 1.5e-8 that a 32-bit sum of two vectors loses: half of the
    # row's mass ends within the first half, 1e-5 before the place where it would end without them
    from paper_2403_10444_b200 import binding as bv
    V, gone = 20480, float("-inf")
    row = torch.full((V // 128, 32, 4), gone)                   # (runs of 32 vectors, two to a sub-segment)
    row[0::2, :, 0] = 0.0
    row[1:V // 256:2, :, 0] = -18.0
    tt = torch.full((V, V), gone, device="cuda")
    tt[0, 7] = 0.0
    tt[7] = row.flatten().cuda()
    dt = torch.full((V, V), gone, device="cuda")
    dt[0, 7] = 0.0
    first = torch.zeros((1,), dtype=torch.int32, device="cuda")
    u = torch.full((1, 1, 3), 0.5, device="cuda")
    tokens = bv.bv_decode_loop(tt, dt, first, u[:, :, :1].contiguous(), u, 1, 1.0, algo)[0]
    assert bv.bv_last_launch_count() == 1
    assert tokens[0].tolist() == [7, V // 2 - 132]
