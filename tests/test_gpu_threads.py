"""Calls from several host threads: two threads issuing calls of different shapes
at once, each on its own stream with its own buffers (the binding releases the
interpreter lock inside a call), and a thread whose first use of the GPU is the
call.  Every call is accepted and every output is bit for bit that of the call
alone."""
import threading

import pytest
import torch

from paper_2509_16686_gb300 import _lib, device, synth

pytestmark = pytest.mark.gpu

CALLS = 6000      # per thread
IN_FLIGHT = 100   # calls issued between two waits for the stream


def step_of(dims, lens):
    dc = device.upload(synth.make_case("threads", dims, lens, seed=81, latent_scale=0.5, layout="permuted"))
    return (lambda stream: dc.bind(stream)), dc.out, dc.status


def prefill_of(d_c):
    dims = synth.Dims(num_heads=2, d_nope=128, d_rope=64, d_v=128, d_c=d_c, page_size=64, vocab=300, dtype="bf16")
    dp = device.upload_prefill(synth.make_prefill_case("threads", dims, [100], seed=82))
    return (lambda stream: lambda: dp.run(stream)), dp.out, dp.status


def r0_of(d_c):
    case = synth.make_case("threads", synth.dims_bf16(d_c=d_c, vocab=300), [70], seed=83, latent_scale=0.5)
    r0 = synth.make_r0_inputs(case, seed=84)
    dc = device.upload(case)
    dc.append()
    w, gate = (device.to_device_array(x, "bf16", "cuda") for x in (r0.w_ukv, r0.gate_r0))
    gamma, beta = torch.from_numpy(r0.gamma).cuda(), torch.from_numpy(r0.beta).cuda()
    ws = torch.empty(_lib.eg_mla_decode_r0_workspace_size(dc.dims, 1, dc.block_table.shape[1], case.num_pages),
                     dtype=torch.uint8, device="cuda")
    out = torch.empty((1, 16, 128), dtype=torch.bfloat16, device="cuda")
    return (lambda stream: lambda: _lib.eg_mla_decode_r0(
        dc.dims, dc.q, dc.c_pool, dc.kr_pool, dc.id_pool, dc.block_table, dc.seq_lens, w, gate, gamma, beta, out, ws,
        dc.status, stream)), out, dc.status


def table_of(d_e):
    dims = _lib.make_dims(16, 128, 64, 128, 128, 300)
    g = torch.Generator(device="cuda").manual_seed(85)
    emb, w_ue = (torch.randn(n, d_e, generator=g, device="cuda").bfloat16() for n in (300, 128))
    out = torch.empty((300, 128), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    return (lambda stream: lambda: _lib.eg_mla_gate_table(dims, emb, w_ue, out, status, stream)), out, status


def fp32_dims(d_c, d_rope):
    return synth.Dims(num_heads=2, d_nope=16, d_rope=d_rope, d_v=16, d_c=d_c, page_size=64, vocab=300, dtype="fp32")


# pairs of calls whose kernels are the same but need different amounts of shared memory
PAIRS = {
    "step_batch": lambda: (step_of(synth.dims_bf16(vocab=300), [70] * 4),
                           step_of(synth.dims_bf16(vocab=300), [70] * 256)),
    "step_width": lambda: (step_of(synth.dims_bf16(d_c=192, vocab=300, gate=False), [70] * 24),
                           step_of(synth.dims_bf16(d_c=512, vocab=300, gate=False), [70] * 12)),
    "step_fp32": lambda: (step_of(fp32_dims(260, 4), [70]), step_of(fp32_dims(512, 64), [70])),
    "prefill": lambda: (prefill_of(64), prefill_of(256)),
    "r0": lambda: (r0_of(192), r0_of(256)),
    "gate_table": lambda: (table_of(64), table_of(256)),
}


@pytest.mark.parametrize("name", sorted(PAIRS))
def test_calls_of_two_threads_leave_each_other_alone(gpu_lib, name):
    work = PAIRS[name]()
    streams = [torch.cuda.Stream() for _ in work]
    calls = [bind(stream) for (bind, _, _), stream in zip(work, streams)]
    torch.cuda.synchronize()
    alone = []
    for call, (_, out, _) in zip(calls, work):
        call()
        torch.cuda.synchronize()
        alone.append(out.clone())
    torch.cuda.synchronize()
    start, errors = threading.Barrier(len(work)), []

    def run(call, stream):
        try:
            torch.cuda.synchronize()   # the device's context is current in this thread
            start.wait()
            for i in range(CALLS):
                call()
                if i % IN_FLIGHT == IN_FLIGHT - 1:
                    stream.synchronize()
        except Exception as e:   # noqa: BLE001 - shown below
            errors.append(e)

    threads = [threading.Thread(target=run, args=a) for a in zip(calls, streams)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    for (_, out, status), want in zip(work, alone):
        assert int(status.item()) == 0
        assert torch.equal(out, want)


@pytest.mark.parametrize("name", sorted(PAIRS))
def test_call_from_a_thread_that_has_used_no_gpu_yet(gpu_lib, name):
    bind, out, status = PAIRS[name]()[0]
    call = bind(torch.cuda.current_stream())
    call()
    want = out.clone()
    out.fill_(0)
    torch.cuda.synchronize()
    errors = []

    def run():
        try:
            call()
        except Exception as e:   # noqa: BLE001 - shown below
            errors.append(e)

    t = threading.Thread(target=run)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert int(status.item()) == 0 and torch.equal(out, want)
