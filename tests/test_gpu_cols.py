"""The weights-as-rows FFN kernel (csrc/gemm_cols.cu): resident and streamed
calls at the edges of its tiles, against the fp64 oracle, and against the
row-major split launches of the same call.

Shapes: tiles of 1 to 128 tokens and several per expert, H and I whose 4-bit
code rows end inside a weight slot, groups without rows, with and without the
shared expert (its group's tiles are bf16 in both weight formats)."""
import numpy as np
import pytest
import torch

import synth
from gpu_case import Case, bf16_bits, bf16_tensor, compare_out, compare_routes
from paper_2608_23805_gb300 import native as N

pytestmark = pytest.mark.gpu


def run_case(tokens, wdtype, streamed, hidden, inter, experts, top_k, shared, residual=False, slots=8):
    cfg = synth.config("tiny", hidden=hidden, inter=inter, n_experts=experts, top_k=top_k, tokens=tokens,
                       n_slots=slots if streamed else experts, wdtype=wdtype, has_shared=shared)
    case = Case(cfg)
    x_bits = synth.hidden(cfg)
    x = bf16_tensor(x_bits)
    ref = case.oracle_layer(x_bits, residual=residual)
    if streamed:
        out, ev = case.plan.forward_streamed(0, x, case.router[0], residual=residual)
    else:
        table, gens = case.stage_all()
        out, ev = case.plan.forward(0, x, case.router[0], table, gens, residual=residual)
        split, _ = case.plan.forward(0, x, case.router[0], table, gens, residual=residual, single_cta=True,
                                     split_waves=True)
    torch.cuda.synchronize()
    assert case.plan.status() == 0
    compare_routes(ev.ids.cpu().numpy(), ev.weights.cpu().numpy(), ref)
    compare_out(bf16_bits(out), ref["out"])
    if not streamed:
        # the same products summed in fp32 over the same K order: outputs
        # differ by no more than a rounding of h and of y
        a, b = out.float(), split.float()
        assert (a - b).norm() <= 2e-3 * b.norm()
    case.close()


@pytest.mark.parametrize("tokens", [1, 2, 15, 17, 33, 64, 129, 500, 700])
@pytest.mark.parametrize("streamed", [False, True])
def test_q4_lengths(tokens, streamed):
    run_case(tokens, synth.W_Q4G32, streamed, 512, 512, 16, 4, not streamed)


@pytest.mark.parametrize("hidden,inter,experts,top_k", [(256, 128, 16, 2), (768, 384, 8, 1), (1024, 640, 24, 8),
                                                        (2048, 512, 64, 10)])
@pytest.mark.parametrize("shared", [False, True])
def test_q4_shapes(hidden, inter, experts, top_k, shared):
    run_case(90, synth.W_Q4G32, False, hidden, inter, experts, top_k, shared, residual=True)


@pytest.mark.parametrize("tokens", [70, 80])
def test_q4_wave_of_all_groups(tokens):
    # one wave of all 32 groups of ~10 rows: more 32-token tiles than a bank
    # of counters may hold
    run_case(tokens, synth.W_Q4G32, True, 512, 256, 32, 4, False, slots=64)


@pytest.mark.parametrize("tokens", [1, 3, 16, 17, 40])
def test_bf16_lengths(tokens):
    run_case(tokens, synth.W_BF16, False, 512, 256, 64, 8, True)


@pytest.mark.parametrize("tokens", [1, 9, 60])
def test_bf16_without_shared_expert(tokens):
    # the kernel's while min(rows, experts) I / 64 fits the SMs
    run_case(tokens, synth.W_BF16, False, 512, 256, 32, 2, False)


@pytest.mark.parametrize("hidden,inter,experts,top_k", [(256, 128, 16, 2), (768, 384, 32, 1), (1024, 640, 64, 8)])
def test_bf16_shapes(hidden, inter, experts, top_k):
    run_case(20, synth.W_BF16, False, hidden, inter, experts, top_k, True)


@pytest.mark.parametrize("wdtype,hidden,inter,experts,top_k,tokens,launches", [
    # the shared expert in the FFN's launch up to 64 rows of a 4-bit layer,
    # else in two of its own
    (synth.W_Q4G32, 512, 128, 16, 2, 64, (1, 0, 0)), (synth.W_Q4G32, 512, 128, 16, 2, 65, (1, 1, 0)),
    # two row-major launches from 24 rows a group of small experts, from 512
    (synth.W_Q4G32, 256, 128, 4, 1, 95, (1, 1, 0)), (synth.W_Q4G32, 256, 128, 4, 1, 96, (0, 1, 1)),
    (synth.W_Q4G32, 512, 512, 4, 1, 2047, (1, 1, 0)), (synth.W_Q4G32, 512, 512, 4, 1, 2048, (0, 1, 1)),
    # a bf16 layer: in the FFN's launch on weights as rows (to 256 rows, 8 a
    # group), else beside the row-major one
    (synth.W_BF16, 256, 128, 64, 1, 256, (1, 0, 0)), (synth.W_BF16, 256, 128, 64, 1, 257, (1, 1, 0)),
    (synth.W_BF16, 256, 128, 16, 4, 32, (1, 1, 0))])
def test_routes(wdtype, hidden, inter, experts, top_k, tokens, launches):
    cfg = synth.config("tiny", hidden=hidden, inter=inter, n_experts=experts, top_k=top_k, tokens=tokens,
                       n_slots=experts, wdtype=wdtype, has_shared=True)
    case = Case(cfg)
    table, gens = case.stage_all()
    x_bits = synth.hidden(cfg)
    case.plan.timing(True)
    out, _ = case.plan.forward(0, bf16_tensor(x_bits), case.router[0], table, gens)
    torch.cuda.synchronize()
    n = {k: v[1] for k, v in case.plan.timing_read().items()}
    assert (n["ffn"], n["shared_gateup"], n["gateup"]) == launches
    compare_out(bf16_bits(out), case.oracle_layer(x_bits)["out"])
    case.close()


@pytest.mark.parametrize("hidden,inter,tokens", [(256, 128, 47), (768, 128, 47), (1280, 640, 60), (1024, 256, 60)])
def test_q4_shared_expert_in_large_tiles(hidden, inter, tokens):
    # 64- and 128-token tiles, and shared and routed tiles of an odd and an even
    # number of weight slots and stages
    run_case(tokens, synth.W_Q4G32, False, hidden, inter, 16, 8, True)


# calls on this kernel with each of its token paths and groups: the shared
# expert inside, 128-token tiles, a wave, bf16 behind the tensor router, bf16
FORMS = [(synth.W_Q4G32, False, 512, 256, 16, 4, 40, True), (synth.W_Q4G32, False, 512, 512, 16, 4, 700, True),
         (synth.W_Q4G32, True, 512, 256, 16, 4, 90, False), (synth.W_BF16, False, 1024, 256, 64, 4, 50, True),
         (synth.W_BF16, False, 256, 128, 64, 1, 200, True)]


def form_case(wdtype, streamed, hidden, inter, experts, top_k, tokens, shared):
    cfg = synth.config("tiny", hidden=hidden, inter=inter, n_experts=experts, top_k=top_k, tokens=tokens,
                       n_slots=8 if streamed else experts, wdtype=wdtype, has_shared=shared)
    case = Case(cfg)
    table = None if streamed else case.stage_all()

    def call(x, out):
        if streamed:
            return case.plan.forward_streamed(0, x, case.router[0], out=out)
        return case.plan.forward(0, x, case.router[0], *table, out=out)

    return cfg, case, call


@pytest.mark.parametrize("form", FORMS)
def test_expired_wait_fails_closed_then_recovers(form):
    # one wait of each launch that nothing ends, with a limit of ~1 ms: the
    # launch gives up, lands its copies and reports a timeout
    cfg, case, call = form_case(*form)
    x_bits = synth.hidden(cfg)
    x = bf16_tensor(x_bits)
    out = torch.full_like(x, 7.0)
    case.plan.set_wait_cycles(2_000_000)
    case.plan.inject(N.MSI_FAULT_DEVICE_WAIT, 0, 0)
    call(x, out)
    torch.cuda.synchronize()
    assert case.plan.status() == N.MSI_ERR_TIMEOUT
    assert torch.all(out == 7.0)
    case.plan.set_wait_cycles(0)
    call(x, out)
    torch.cuda.synchronize()
    assert case.plan.status() == N.MSI_OK
    compare_out(bf16_bits(out), case.oracle_layer(x_bits)["out"])
    case.close()


@pytest.mark.parametrize("kind,status", [(N.MSI_FAULT_STALE_COMPLETION, N.MSI_ERR_STALE_GENERATION),
                                         (N.MSI_FAULT_WRONG_OBJECT, N.MSI_ERR_WRONG_OBJECT)])
@pytest.mark.parametrize("form", [FORMS[0], FORMS[2]])
def test_wrong_publication_fails_closed(form, kind, status):
    # a slot whose published word is not the plan's: the launch (a wave), or the
    # scatter before it, rejects its group and no row becomes visible
    streamed = form[1]
    cfg, case, call = form_case(*form)
    x_bits = synth.hidden(cfg)
    x = bf16_tensor(x_bits)
    used = np.unique(case.oracle_layer(x_bits)["ids"])
    out = torch.full_like(x, 5.0)
    e = int(used[len(used) // 2])
    case.plan.inject(kind, 0, e)
    if not streamed:
        case.plan.stage(e, 0, e)
        gens = case.plan.slot_table(0)
        case.plan.forward(0, x, case.router[0], *gens, out=out)
    else:
        call(x, out)
    torch.cuda.synchronize()
    assert case.plan.status() == status
    assert torch.all(out == 5.0)
    case.close()


@pytest.mark.parametrize("form", FORMS)
def test_back_to_back_calls_on_one_workspace(form):
    # four chained calls with other inputs, nothing waited for between them:
    # each output is that of the same call alone
    cfg, case, call = form_case(*form)
    xs = [bf16_tensor(synth.hidden(cfg, 0, i)) for i in range(4)]
    outs = [torch.empty_like(x) for x in xs]
    for x, out in zip(xs, outs):
        call(x, out)
    torch.cuda.synchronize()
    assert case.plan.status() == N.MSI_OK
    for x, out in zip(xs, outs):
        alone = torch.empty_like(x)
        call(x, alone)
        torch.cuda.synchronize()
        assert torch.equal(out.view(torch.int16), alone.view(torch.int16))
    compare_out(bf16_bits(outs[3]), case.oracle_layer(synth.hidden(cfg, 0, 3))["out"])
    case.close()
