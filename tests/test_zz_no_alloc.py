"""The entry point that allocates nothing (ouro_lm_head_static).

Collected last on purpose: if it fails, a run that stops at the first failure has already run everything else.
Who needs it: users of this library who cannot hand it a workspace or let it allocate - a serving process whose
own arena owns all device memory, or a loop that must not risk the synchronisation an allocation can cause.  The
call keeps the GEMM's split-K scratch in a fixed 5 MiB array inside the library instead.

Expected values, first: logits = x . lm_head^T evaluated in float64 by numpy on the very bf16 inputs the call
gets (the definition of the LM-head pass, nothing of the CUDA path in it).  Second, as a cross-check between the
two entry points: a one-layer model whose output projections are zero leaves the residual stream equal to the
token embeddings, so the regular ouro_verify_forward computes logits = normalise(embedding rows) x lm_head^T; the
static call gets the same normalised rows and the same head and must agree to bf16 rounding.

Shapes are chosen so that the static array's split-K slots and counters are really used: with 32 CTAs a
vocabulary of 4000 (32 tiles) takes only whole tiles, 2048 (16 tiles) splits every tile between two CTAs, 4104
(33 tiles) leaves one ragged tile of 8 entries cut four ways, and a 64-wide model leaves fewer work items than
CTAs.  Every shape is run twice in a row with different rows, so a counter or a slot left over from the
previous call would show.
"""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_2402_13720_b200 import binding, build, synth

pytestmark = pytest.mark.gpu
BF16_REL = 3e-2     # same bound as the parity tests: per row, relative to the largest |logit|


def _verify_forward_logits(desc, w, tokens):
    P = synth.DecodeParams(2, 3, 1, 4, 4, seed_prompt=False)
    eng = binding.Engine(desc, w, P)
    eng.assemble_causal(binding.OURO_TARGET, tokens)
    am, lg = eng.verify_forward(want_logits=True)
    torch.cuda.synchronize()
    out = am[: len(tokens)].clone(), lg[: len(tokens)].clone()
    eng.close()
    return out


def _check_against_definition(x, head, arg, logits):
    want = x.double().cpu().numpy() @ head.double().cpu().numpy().T            # float64, the definition
    got = logits.double().cpu().numpy()
    err = np.abs(got - want).max(axis=1)
    scale = np.abs(want).max(axis=1)
    assert (err <= BF16_REL * scale).all(), float((err / scale).max())
    srt = np.sort(want, axis=1)
    safe = (srt[:, -1] - srt[:, -2]) > 2 * err + 1e-9
    assert safe.sum() >= 1 and np.array_equal(arg.cpu().numpy()[safe], want.argmax(axis=1)[safe])
    assert torch.equal(arg.long(), logits.argmax(dim=1))                       # consistent with its own logits
    return err


@pytest.mark.parametrize("d_model,vocab", [(256, 4000), (256, 2048), (256, 4104), (64, 2048), (512, 1032)])
def test_static_scratch_head_equals_the_definition_twice(d_model, vocab):
    build.build()
    head = synth.tensor(21, 3, (vocab, d_model), 0.02, torch.bfloat16, "cuda:0")
    for call, rows in enumerate((37, 5, 128)):                                 # calls in a row, different sizes
        x = synth.tensor(22 + call, 4, (rows, d_model), 1.0, torch.bfloat16, "cuda:0")
        arg, logits = binding.lm_head_static(x, head, want_logits=True)
        _check_against_definition(x, head, arg, logits)
        arg2, _ = binding.lm_head_static(x, head)                              # without logits: same greedy tokens
        assert torch.equal(arg2, arg)


@pytest.mark.parametrize("d_model,vocab", [(64, 18944), (192, 19080), (128, 23048), (128, 23176), (64, 65536)])
def test_static_scratch_head_over_all_sms(d_model, vocab):
    """More whole tiles than one CTA per SM (148) takes at once, beside 20, 22, 21, 22 and no tiles that the CTAs with slots
    share: 148 tiles, 150 and 181 with a ragged last one, 182, and the largest vocabulary (512)."""
    build.build()
    head = synth.tensor(41, 3, (vocab, d_model), 0.02, torch.bfloat16, "cuda:0")
    for call, rows in enumerate((1, 37, 128)):
        x = synth.tensor(42 + call, 4, (rows, d_model), 1.0, torch.bfloat16, "cuda:0")
        arg, logits = binding.lm_head_static(x, head, want_logits=True)
        _check_against_definition(x, head, arg, logits)
        few, _ = binding.lm_head_static(x[:1].contiguous(), head)
        assert torch.equal(few, arg[:1])                         # a row's choice does not depend on the others


def test_static_scratch_head_keeps_the_precision_of_its_cut_tiles():
    """250 tiles of 4096 columns: 26 are summed along K in pieces (the remainder of a launch over the 32 CTAs that have
    slots), the others in one chain.  The pieces' sum is nearer to the exact one, so a launch that handled the remainder
    whole would show it: the error of those columns against float64 would equal that of the others (measured: 0.75 of it)."""
    build.build()
    d_model, vocab, rows = 4096, 32000, 37
    x = synth.tensor(51, 4, (rows, d_model), 1.0, torch.bfloat16, "cuda:0")
    head = synth.tensor(52, 3, (vocab, d_model), 0.02, torch.bfloat16, "cuda:0")
    _, logits = binding.lm_head_static(x, head, want_logits=True)
    err = torch.cat([logits[:, a: a + 4000].double() - x.double() @ head[a: a + 4000].double().T for a in range(0, vocab, 4000)], 1)
    cut = (vocab // 128 - 26) * 128
    whole, pieces = (float(e.square().mean().sqrt()) for e in (err[:, :cut], err[:, cut:]))
    assert pieces < 0.9 * whole, (pieces, whole)


def test_static_scratch_head_matches_verify_forward_twice():
    build.build()
    desc = synth.ModelDesc(1, 256, 4, 4, 64, 256, 4104, 192, "bf16")
    w = synth.model_weights(desc, 11, device="cuda:0")
    w["layers"][0]["wo"].zero_()
    w["layers"][0]["w_down"].zero_()
    rng = np.random.default_rng(0)
    for call, rows in enumerate((37, 5)):                       # two calls in a row, different sizes
        tokens = rng.integers(0, desc.vocab, rows).astype(np.int32)
        ref_arg, ref_logits = _verify_forward_logits(desc, w, tokens)
        x = w["embed"][torch.as_tensor(tokens.astype(np.int64), device="cuda:0")].float()
        inv = 1.0 / torch.sqrt((x * x).mean(dim=1, keepdim=True) + desc.rms_eps)
        xn = (w["final_norm"].float() * (x * inv)).to(torch.bfloat16).contiguous()
        arg, logits = binding.lm_head_static(xn, w["lm_head"], want_logits=True)
        _check_against_definition(xn, w["lm_head"], arg, logits)
        err = (logits - ref_logits).abs().amax(dim=1)
        scale = ref_logits.abs().amax(dim=1)
        assert bool((err <= BF16_REL * scale).all()), (call, float((err / scale).max()))
        top2 = ref_logits.topk(2, dim=1).values
        safe = (top2[:, 0] - top2[:, 1]) > 2 * err + 1e-6
        assert int(safe.sum()) >= 1 and torch.equal(arg[safe], ref_arg[safe])


def test_static_scratch_is_left_clear_whatever_a_call_finds_in_it():
    """Calls that overlap on a device race on the array, which the header forbids; what they leave there must not reach a
    later call.  Stand-in for such leftovers: the slots filled by hand.  The call that meets them may be wrong, but it leaves
    no partial sum behind, and the next one gives the bits of the first.  A raised status word is reported once."""
    build.build()
    head = synth.tensor(61, 3, (2048, 256), 0.02, torch.bfloat16, "cuda:0")
    x = synth.tensor(62, 4, (37, 256), 1.0, torch.bfloat16, "cuda:0")
    want = binding.lm_head_static(x, head, want_logits=True)
    ptr, nbytes = C.c_void_p(), C.c_size_t()
    assert binding.lib().ouro_debug_static_scratch(C.byref(ptr), C.byref(nbytes)) == binding.OURO_OK

    class Scratch:
        __cuda_array_interface__ = dict(shape=(nbytes.value // 4 + 1,), typestr="<i4", data=(ptr.value, False), version=2)

    words = torch.as_tensor(Scratch(), device="cuda:0")
    slots, status = words[:-1].view(-1, 128 * 128), words[-1:]
    assert bool((slots == -1).all()) and int(status[0]) == 0
    for garbage in (0, 0x3F800000):
        slots[:, : 37 * 128] = garbage
        torch.cuda.synchronize()
        binding.lm_head_static(x, head)
        assert bool((slots == -1).all()) and int(status[0]) == 0
        got = binding.lm_head_static(x, head, want_logits=True)
        assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    status[0] = 1                                                # a give-up of another call: reported once, then gone
    torch.cuda.synchronize()
    with pytest.raises(binding.OuroError):
        binding.lm_head_static(x, head)
    got = binding.lm_head_static(x, head, want_logits=True)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])


def test_static_scratch_head_breaks_exact_ties_towards_the_smallest_id():
    """Identical rows of the head give bit-identical logits; the greedy choice must then be the smallest id,
    whether the copies share a 128-entry tile or not."""
    build.build()
    d_model, vocab = 256, 2048
    head = synth.tensor(31, 3, (vocab, d_model), 0.02, torch.bfloat16, "cuda:0")
    x = synth.tensor(32, 4, (37, d_model), 1.0, torch.bfloat16, "cuda:0")
    win = (x[0].float() * 0.05).to(torch.bfloat16)               # a row whose logit for x[0] dominates
    for ids in ((700, 731, 1500), (1990, 130, 131)):
        h = head.clone()
        for i in ids:
            h[i] = win
        arg, logits = binding.lm_head_static(x, h, want_logits=True)
        assert len({float(logits[0, i]) for i in ids}) == 1 and int(logits[0].argmax()) in ids
        assert int(arg[0]) == min(ids)


def test_static_scratch_rejects_sizes_beyond_its_limits():
    build.build()
    x = torch.zeros((4, 128), dtype=torch.bfloat16, device="cuda:0")
    big = torch.zeros((8, 128), dtype=torch.bfloat16, device="cuda:0")
    lib = binding.lib()
    am = torch.zeros(4, dtype=torch.int32, device="cuda:0")
    rc = lib.ouro_lm_head_static(x.data_ptr(), big.data_ptr(), 4, 128, 65536 + 8, am.data_ptr(), None, None)
    assert rc == binding.OURO_EINVAL and b"static scratch" in lib.ouro_last_error(None)
    assert lib.ouro_lm_head_static(x.data_ptr(), big.data_ptr(), 129, 128, 8, am.data_ptr(), None, None) == binding.OURO_EINVAL
    assert lib.ouro_lm_head_static(x.data_ptr(), big.data_ptr(), 4, 100, 8, am.data_ptr(), None, None) == binding.OURO_EINVAL
