"""The pruning step's compaction starting before the selection has read the head
scores: outputs that share memory with Q or with the workspace, a call of each
kind after the other on one workspace and one set of outputs, against a call with
buffers of its own."""
import pytest
import torch

from paper_2608_25332_gb300 import provip as P
from paper_2608_25332_gb300 import synth

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    import __graft_entry__
    __graft_entry__.build()
    yield
    rc, bits = P.provip_device_status(clear=True)
    assert rc == 0 and bits == 0, f"device status {rc} {bits}"


def case(name):
    w = synth.BY_NAME[name]
    cpu = synth.in_llm_inputs(w)
    return w, {k: (v.to(DEV) if isinstance(v, torch.Tensor) else v) for k, v in cpu.items()}


def call(step, g, Q=None):
    step(g["Q"] if Q is None else Q, g["K"], g["V"], g["hidden"], g["pos"], g["text_start"], g["text_len"],
         g["seq_len"], g["vis_start"])


def outputs(step, w):
    n = step.seq_len_out.tolist()
    rows = [torch.cat([t[b, :n[b]].reshape(-1) for b in range(w.B)]) for t in
            (step.hidden_out, step.K_out, step.V_out)]
    pos = torch.cat([step.pos_out[:, b, :n[b]].reshape(-1) for b in range(w.B)])
    return [t.clone().view(torch.int16) if t.dtype == torch.bfloat16 else t.clone()
            for t in (*rows, pos, step.idx, step.seq_len_out, step.scores)]


@pytest.mark.parametrize("name,algo", [("llava15_7b_bf16_b16", P.ALGO_AUTO), ("llava_next_7b_bf16_b8", P.ALGO_AUTO),
                                       ("llava_next_7b_bf16_b8", P.ALGO_TCGEN05_STREAM),
                                       ("video_gqa_bf16_b1", P.ALGO_TCGEN05_TWOPASS),
                                       ("llava15_7b_f32_b1", P.ALGO_AUTO)])
def test_outputs_in_the_memory_of_q_or_the_workspace(name, algo):
    w, g = case(name)
    make = lambda **k: P.PruneStep(g["Q"], g["K"], g["V"], g["hidden"], g["pos"], g["head_list"], w.n_t[1], g["N_v"],
                                   w.keep, algo=algo, **k)
    own = make()
    call(own, g)
    torch.cuda.synchronize()
    ref = outputs(own, w)
    step = make()
    for turn in range(4):
        Q = g["Q"].clone()
        n = step.hidden_out.numel()
        if turn % 2 == 0:  # the hidden states go where the queries were
            step.hidden_out = Q.reshape(-1)[:n].view(own.hidden_out.shape)
        else:              # and where the workspace ends
            need = step.ws.numel()
            size = need + n * Q.element_size()
            big = P.workspace(size, DEV)
            step.ws = big
            step.hidden_out = big[need:need + n * Q.element_size()].view(Q.dtype).view(own.hidden_out.shape)
        call(step, g, Q)
        torch.cuda.synchronize()
        for x, y in zip(outputs(step, w), ref):
            assert torch.equal(x, y), (name, turn)


@pytest.mark.parametrize("name", ["llava15_7b_bf16_b16", "video_gqa_bf16_b1"])
def test_calls_of_each_kind_in_turn(name):
    """Plain, overlapping and concurrent calls back to back on one workspace and
    one set of outputs, each on other inputs, then the last one's outputs."""
    w, g = case(name)
    other = dict(g, Q=g["Q"].flip(0).contiguous() if w.B > 1 else -g["Q"])
    kinds = (0, P.PRUNE_OVERLAP_PREVIOUS, 0, P.PRUNE_CONCURRENT, P.PRUNE_OVERLAP_PREVIOUS, 0, 0)
    make = lambda: P.PruneStep(g["Q"], g["K"], g["V"], g["hidden"], g["pos"], g["head_list"], w.n_t[1], g["N_v"],
                               w.keep)
    refs = []
    for x in (g, other):
        s = make()
        call(s, x)
        torch.cuda.synchronize()
        refs.append(outputs(s, w))
    step = make()
    for last in range(1, len(kinds) + 1):
        torch.cuda.synchronize()
        for i, flags in enumerate(kinds[:last]):
            step.flags = flags
            call(step, g if i % 2 == 0 else other)
        torch.cuda.synchronize()
        for x, y in zip(outputs(step, w), refs[(last - 1) % 2]):
            assert torch.equal(x, y), (name, last)
