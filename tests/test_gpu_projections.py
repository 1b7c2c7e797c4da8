"""The fused layer projections and the prompt attention at the sizes where their tiles end: a prompt fed in chunks through
the tensor-core kernels, and a decoder step of many rows, against the same work one kernel per operation (each of the two is
within the bound that holds against the oracle, so they differ by at most twice that bound)."""
import dataclasses

import numpy as np
import pytest
import torch

from paper_2601_20357_b200 import workloads as W

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    import gpu_harness as H
    from paper_2601_20357_b200 import binding as TB


def _workload(B, m, heads, kv_heads, hd, ffn, cap):
    cfg = W.DrafterCfg(2, heads * hd, heads, kv_heads, ffn, 1003, "bf16")
    return W.Workload(name=f"proj{heads}x{hd}", config_id=91, drafter=cfg, n_inputs=m, n_requests=B, gamma=2, window_h=4, rounds=1,
                      policy=W.POLICY_STATIC, prefixes=((("tokens", 1),),) * m, kv_capacity=cap, alpha=(1.0 / m,) * m)


def _handle(wl, weights):
    return TB.Tabed(n_inputs=wl.n_inputs, n_requests=wl.n_requests, gamma=wl.gamma, window_h=wl.window_h, policy=wl.policy,
                    vocab=wl.drafter.vocab, drafter=wl.drafter, weights=weights, kv_capacity=wl.kv_capacity)


def _logits_after(wl, weights, path, lengths, seed):
    """Logits of one decoder step after every row's prompt (token part, then embedding part) has been fed on `path`."""
    g = _handle(wl, weights)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    g.select_path(path)
    for row, (n_tok, n_emb) in enumerate(lengths):
        if n_tok:
            g.prefill_tokens(row, torch.randint(0, wl.drafter.vocab, (n_tok,), generator=gen, device="cuda", dtype=torch.int32))
        if n_emb:
            g.prefill_embeds(row, torch.randn((n_emb, wl.drafter.d_model), generator=gen, device="cuda"))
    tok = torch.randint(0, wl.drafter.vocab, (wl.n_requests,), generator=gen, device="cuda", dtype=torch.int32)
    out = torch.empty((wl.n_rows, wl.drafter.vocab), device="cuda")
    g.decode_step(tok, out)
    torch.cuda.synchronize()
    assert g.last_device_error() == 0
    g.destroy()
    return out.cpu().numpy()


@pytest.mark.parametrize("heads,kv_heads,hd,ffn", [(4, 4, 64, 640), (7, 1, 64, 520), (11, 11, 32, 704), (3, 3, 128, 776)])
@pytest.mark.parametrize("lengths", [((1, 0), (63, 1), (64, 65)), ((0, 129), (255, 2), (1030, 0))])
def test_prompt_chunks_agree_with_one_position_at_a_time(heads, kv_heads, hd, ffn, lengths):
    wl = _workload(1, 3, heads, kv_heads, hd, ffn, 1040)
    weights = TB.weights_to_device(wl.drafter, W.make_weights(wl), torch.device("cuda", 0))
    a = _logits_after(wl, weights, TB.PATH_TENSOR_CORE, lengths, 5)
    b = _logits_after(wl, weights, TB.PATH_PER_OP, lengths, 5)
    assert np.max(np.abs(a - b)) <= 2 * H.logit_tols(wl)[0]


@pytest.mark.parametrize("heads,hd,ffn,n", [(8, 128, 4096, 800), (8, 64, 2560, 700)])
def test_long_prompts_of_wide_drafters_agree_with_one_position_at_a_time(heads, hd, ffn, n):
    """The forms that only much work takes: a kernel of its own per epilogue; 64 positions a CTA of the prompt attention at a
    head size of 128; and, at 1024 / 4096 columns and 800 positions, a down projection whose CTAs read one another's partial
    sums where they lie (tests/test_proj_plan.py checks that the plan is such a one)."""
    wl = _workload(1, 1, heads, heads, hd, ffn, n + 8)
    weights = TB.weights_to_device(wl.drafter, W.make_weights(wl), torch.device("cuda", 0))
    a = _logits_after(wl, weights, TB.PATH_TENSOR_CORE, ((n, 0),), 7)
    b = _logits_after(wl, weights, TB.PATH_PER_OP, ((n, 0),), 7)
    assert np.max(np.abs(a - b)) <= 2 * H.logit_tols(wl)[0]


@pytest.mark.parametrize("B,m", [(1, 1), (5, 3), (11, 3), (43, 3), (129, 2)])
def test_rows_at_tile_edges_agree_with_per_operation_step(B, m):
    """1, 15, 33, 129 and 258 rows: one tile and several, whole and ragged (the plan of a projection depends on the count)."""
    wl = _workload(B, m, 6, 2, 64, 520, 40)
    weights = TB.weights_to_device(wl.drafter, W.make_weights(wl), torch.device("cuda", 0))
    lengths = [(1 + r % 7, 0) for r in range(wl.n_rows)]
    a = _logits_after(wl, weights, TB.PATH_TENSOR_CORE, lengths, 6)
    b = _logits_after(wl, weights, TB.PATH_PER_OP, lengths, 6)
    assert np.max(np.abs(a - b)) <= 2 * H.logit_tols(wl)[0]


@pytest.mark.parametrize("path", [TB.PATH_AUTO, TB.PATH_TENSOR_CORE] if torch.cuda.is_available() else [])
@pytest.mark.parametrize("heads,kv_heads,hd", [(5, 1, 64), (5, 5, 64), (10, 10, 32)])
def test_a_request_that_is_not_finite_leaves_the_others_alone(heads, kv_heads, hd, path):
    """320 columns end in the middle of an operand block.  What the blocks hold there must not come from another slot: the
    prompts, the decoder step and its LM head cut the same buffer differently, so the values of a request whose embeddings
    are NaN lie under every part of the layouts that follow.  The other request's logits keep their bits."""
    wl = _workload(2, 3, heads, kv_heads, hd, 640, 400)
    weights = TB.weights_to_device(wl.drafter, W.make_weights(wl), torch.device("cuda", 0))
    gen = torch.Generator(device="cuda").manual_seed(9)
    emb = [torch.randn((n, wl.drafter.d_model), generator=gen, device="cuda") for n in (37, 130, 5, 300, 64, 129)]
    tok = torch.randint(0, wl.drafter.vocab, (2,), generator=gen, device="cuda", dtype=torch.int32)
    seen = []
    for bad in (False, True):
        g = _handle(wl, weights)
        g.select_path(path)
        for row in (3, 0, 4, 1, 5, 2):
            g.prefill_embeds(row, torch.full_like(emb[row], float("nan")) if bad and row >= 3 else emb[row])
        out = torch.empty((2, wl.n_rows, wl.drafter.vocab), device="cuda")
        for i in range(2):
            g.decode_step(tok, out[i])
        torch.cuda.synchronize()
        seen.append(out[:, :3].cpu().numpy())
        assert np.isfinite(seen[-1]).all()
        assert not bad or not np.isfinite(out[:, 3:].cpu().numpy()).any()
        g.destroy()
    assert np.array_equal(seen[0], seen[1])


@pytest.mark.parametrize("heads,kv_heads,hd", [(8, 4, 32), (2, 1, 128)])
def test_a_prompt_does_not_see_what_a_longer_one_left_in_the_cache(heads, kv_heads, hd):
    """The cache beyond a prompt's last position may still hold an earlier conversation of the row, and that need not have
    been finite: after the saved state is restored, the logits of a shorter prompt have the bits of a fresh handle."""
    wl = _workload(1, 3, heads, kv_heads, hd, 640, 200)
    weights = TB.weights_to_device(wl.drafter, W.make_weights(wl), torch.device("cuda", 0))
    gen = torch.Generator(device="cuda").manual_seed(10)
    emb = [torch.randn((n, wl.drafter.d_model), generator=gen, device="cuda") for n in (17, 65, 100)]
    tok = torch.randint(0, wl.drafter.vocab, (1,), generator=gen, device="cuda", dtype=torch.int32)
    seen = []
    for used in (False, True):
        g = _handle(wl, weights)
        saved = g.state_export()
        if used:
            for row in range(3):
                g.prefill_embeds(row, torch.full((190, wl.drafter.d_model), float("nan"), device="cuda"))
            g.state_import(saved)
        for row in range(3):
            g.prefill_embeds(row, emb[row])
        out = torch.empty((wl.n_rows, wl.drafter.vocab), device="cuda")
        g.decode_step(tok, out)
        torch.cuda.synchronize()
        seen.append(out.cpu().numpy())
        g.destroy()
    assert np.isfinite(seen[1]).all() and np.array_equal(seen[0], seen[1])


def test_more_slot_counts_than_the_table_of_plans_holds():
    """A prompt fed in 22 pieces of 20 different lengths (the table has 16 places), against one position at a time."""
    wl = _workload(1, 1, 4, 2, 64, 640, 240)
    weights = TB.weights_to_device(wl.drafter, W.make_weights(wl), torch.device("cuda", 0))
    gen = torch.Generator(device="cuda").manual_seed(11)
    tok = torch.randint(0, wl.drafter.vocab, (214,), generator=gen, device="cuda", dtype=torch.int32)
    seen = []
    for path in (TB.PATH_TENSOR_CORE, TB.PATH_PER_OP):
        g = _handle(wl, weights)
        g.select_path(path)
        at = 0
        for n in (*range(1, 21), 1, 2):
            g.prefill_tokens(0, tok[at:at + n].contiguous())
            at += n
        out = torch.empty((1, wl.drafter.vocab), device="cuda")
        g.decode_step(tok[at:at + 1].contiguous(), out)
        torch.cuda.synchronize()
        seen.append(out.cpu().numpy())
        g.destroy()
    assert np.max(np.abs(seen[0] - seen[1])) <= 2 * H.logit_tols(wl)[0]


def test_attention_of_a_capacity_beyond_2_to_the_20_takes_the_same_kernel():
    """Row and position of a slot share a word in the attention kernel; more than 2^20 positions fit too."""
    seen = []
    for cap in (300, (1 << 20) + 9):
        wl = _workload(1, 3, 2, 1, 64, 256, cap)
        wl = dataclasses.replace(wl, drafter=dataclasses.replace(wl.drafter, n_layers=1))
        weights = TB.weights_to_device(wl.drafter, W.make_weights(wl), torch.device("cuda", 0))
        g = _handle(wl, weights)
        gen = torch.Generator(device="cuda").manual_seed(12)
        for row, n in enumerate((1, 127, 260)):
            g.prefill_tokens(row, torch.randint(0, wl.drafter.vocab, (n,), generator=gen, device="cuda", dtype=torch.int32))
        before, out = g.launch_count(), torch.empty((wl.n_rows, wl.drafter.vocab), device="cuda")
        g.decode_step(torch.tensor([5], dtype=torch.int32, device="cuda"), out)
        torch.cuda.synchronize()
        seen.append((g.launch_count() - before, out.cpu().numpy()))
        g.destroy()
    assert seen[0][0] == seen[1][0] and np.array_equal(seen[0][1], seen[1][1])
