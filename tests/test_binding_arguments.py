"""What the Python binding refuses and takes before any launch: ranks of the tensors, kinds of numbers.  No GPU is needed: a
call whose shapes are right ends at the check that its tensors lie on the device."""
import pytest
import torch

BF, F32, I32, U8 = torch.bfloat16, torch.float32, torch.int32, torch.uint8
B, HQ, HKV, D, PAGES, P = 2, 4, 2, 128, 5, 16
RIGHT = "CUDA tensor"          # the right shapes on the wrong device


def _context():
    from paper_2512_05033_b200 import build
    build.build()
    from paper_2512_05033_b200 import binding
    c = binding.Context.__new__(binding.Context)   # no arb_ctx: nothing gets as far as using one
    c._h = c._p = None
    return c, binding


def _t(*shape, dtype=BF):
    return torch.zeros(*shape, dtype=dtype)


def _args():
    q, rows = _t(B, HQ, D), _t(B, HKV, D)
    pool, codes, half = _t(PAGES, HKV, P, D), _t(PAGES, HKV, P, D, dtype=U8), _t(PAGES, HKV, P, D // 2, dtype=U8)
    sc, table, lens = _t(PAGES, HKV, P, dtype=F32), _t(B, 3, dtype=I32), _t(B, dtype=I32)
    s4 = (1.0, 1.0, 1.0, 1.0)
    # entry point -> (positional arguments, {argument: rank asked for})
    return {
        "attn": ([q, pool, pool, table, lens, lens, 1], {0: 3, 1: 4, 3: 2}),
        "decode_step": ([q, rows, rows, pool, pool, table, lens, lens], {0: 3, 3: 4, 5: 2}),
        "decode_step_e4m3": ([q, rows, rows, codes, codes, *s4, table, lens, lens], {0: 3, 3: 4, 9: 2}),
        "decode_step_i4": ([q, rows, rows, half, half, sc, sc, table, lens, lens], {3: 4, 7: 2}),
        "attn_decode_e4m3": ([q, codes, codes, 1.0, 1.0, table, lens, lens], {0: 3, 1: 4, 5: 2}),
        "attn_e4m3": ([q, codes, codes, 1.0, 1.0, table, lens, lens, 1], {0: 3, 1: 4, 5: 2}),
        "kv_append": ([rows, rows, table, lens, lens, pool, pool], {2: 2, 5: 4}),
        "kv_append_e4m3": ([rows, rows, 1.0, 1.0, table, lens, lens, codes, codes], {4: 2, 7: 4}),
        "kv_append_i4": ([rows, rows, table, lens, lens, half, half, sc, sc], {2: 2, 5: 4}),
        "route": ([_t(3, 64), _t(64), 0.0, 0.5], {0: 2}),
        "route_classes": ([0, _t(3, 64), _t(2, 64), [0.0, 0.0], 0.5], {1: 2}),
    }


@pytest.mark.parametrize("name", list(_args()))
def test_wrong_ranks_are_refused(name):
    c, _ = _context()
    args, ranks = _args()[name]
    with pytest.raises(ValueError, match=RIGHT):
        getattr(c, name)(*args)
    for i, rank in ranks.items():
        for bad in (args[i][None], args[i][0]):
            with pytest.raises(ValueError, match=f"must have {rank} dimensions"):
                getattr(c, name)(*args[:i], bad, *args[i + 1:])


def test_host_calls_refuse_wrong_ranks():
    c, _ = _context()
    q, pool, table, lens = _t(B, HQ, D), _t(PAGES, HKV, P, D), _t(B, 3, dtype=I32), _t(B, dtype=I32)
    for call in (lambda *a: c.attn_host(*a, lens, lens, 1, out_host=q), lambda *a: c.attn_host_begin(*a, lens, lens, 1, q)):
        with pytest.raises(ValueError, match=RIGHT):
            call(q, pool, pool, table)
        for a, rank in (((q[None], pool, pool, table), 3), ((q, pool[None], pool, table), 4), ((q, pool, pool, table[0]), 2)):
            with pytest.raises(ValueError, match=f"must have {rank} dimensions"):
                call(*a)


def test_a_record_of_parameters_leaves_the_shapes_to_the_caller():
    c, binding = _context()
    p = binding.attn_params(binding.ARB_BF16, B, HQ, HKV, D, PAGES, 3, B, 1)
    pool, table, lens = _t(PAGES * HKV * P, D), _t(B * 3, dtype=I32), _t(B, dtype=I32)
    with pytest.raises(ValueError, match=RIGHT):
        c.attn(_t(B, HQ * D), pool, pool, table, lens, lens, 1, params=p)
    with pytest.raises(ValueError, match=RIGHT):
        c.decode_step(_t(B, HQ * D), _t(B, HKV * D), _t(B, HKV * D), pool, pool, table, lens, lens, params=p)


def test_numbers_are_taken_as_int_and_float_take_them():
    c, binding = _context()
    scores, lens = _t(4, dtype=F32), _t(B, dtype=I32)
    with pytest.raises(ValueError, match=RIGHT):
        c.policy(binding.POLICY_ORACLE_BUDGET, scores, scores, tau=torch.tensor(0.5), budget=2.0)
    with pytest.raises(ValueError, match=RIGHT):
        c.phase_lens(lens, want=1.0, t=0.0)
    with pytest.raises(ValueError, match=RIGHT):
        c.phase_lens_tokens(lens, 3, want=True)
    with pytest.raises(TypeError):
        c.attn(_t(B, HQ, D), _t(PAGES, HKV, P, D), _t(PAGES, HKV, P, D), _t(B, 3, dtype=I32), lens, lens, 1.0)


def test_the_extension_module_is_built_again_for_another_interpreter_or_torch(monkeypatch):
    from paper_2512_05033_b200 import build
    build.build()
    assert not build.native_stale()
    monkeypatch.setattr(build, "_native_abi", lambda: "python 3.99\ntorch 9.9\n")
    assert build.native_stale()


@pytest.mark.gpu
def test_a_negative_number_of_tokens_is_refused():
    from tests import helpers as H
    from paper_2512_05033_b200 import binding
    lens, out = torch.full((B,), 3, dtype=I32, device="cuda"), torch.full((B,), 77, dtype=I32, device="cuda")
    with pytest.raises(binding.ArbError):
        H.ctx().phase_lens_tokens(lens, -1, out=out)
    assert H.ctx().poll_status() == 0 and bool((out == 77).all())
