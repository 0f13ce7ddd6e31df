"""Prefiltering and lighting sets by several threads at once, on streams of their own, with unequal needs
of shared memory (rows staged in shared memory, rows read through L1, wide and narrow irradiance
pieces): every call succeeds and every output has the bits of the call made alone."""
import ctypes as C
import threading

import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2012_03325_gb300 as ep  # noqa: E402

THREADS, CALLS = 4, 1500


def outputs(ibl, levels):
    return [ibl.level(m).clone() for m in range(levels)] + [ibl.irradiance().clone(), ibl.lut().clone()]


# (width, height, levels, samples) of the threads' environments, in turn
@pytest.mark.parametrize("whole_set,a,b", [(False, (256, 2, 3, 2000), (256, 2, 3, 4)),
                                           (False, (100, 8, 4, 2000), (100, 8, 4, 8)),
                                           (True, (2048, 2, 1, 4), (64, 2, 1, 4))])
def test_threads(whole_set, a, b):
    jobs, failures = [], []
    for q in range(THREADS):
        We, He, M, N = b if q % 2 else a
        env = torch.from_numpy(synth.make_env(12 + q, We, He)).cuda()
        p = ep.ibl_params(M, N, 8, 8, 4, 2)
        ibl = ep.Ibl(p, We, He)
        ws = torch.empty(ep.epbr_precompute_ibl_workspace_size(p, We, He) + 512, dtype=torch.uint8, device="cuda")
        ep.epbr_precompute_ibl(env, ibl, workspace=ws)
        want = outputs(ibl, M)
        for m in range(M):
            ibl.level(m).zero_()
        jobs.append((env, p, ibl, ws, M, want, torch.cuda.Stream()))
    torch.cuda.synchronize()
    start = threading.Barrier(THREADS, timeout=60)

    def work(env, p, ibl, ws, M, want, stream):
        e, base = ep.env_struct(env), (ws.data_ptr() + 255) & ~255
        room, lib = ws.numel() - (base - ws.data_ptr()), ep.lib()
        start.wait()
        for k in range(CALLS):
            if whole_set:
                st = lib.epbr_precompute_ibl(C.byref(e), C.byref(p), C.byref(ibl.struct), base, room, stream.cuda_stream)
            else:
                st = lib.epbr_prefilter(C.byref(e), p.prefilter_samples, C.byref(ibl.struct), stream.cuda_stream)
            if st:
                failures.append((k, st))
            if k % 20 == 19:  # the streams' queues stay short, so that the threads meet in the calls
                stream.synchronize()

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failures, (len(failures), failures[:4])
    for env, p, ibl, ws, M, want, stream in jobs:
        for g, w in zip(outputs(ibl, M), want):
            assert torch.equal(g, w)
