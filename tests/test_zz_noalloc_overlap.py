"""tune_eval_noalloc with TUNE_EMIT_POINTS from several host threads, each on a stream of its own: the calls
overlap on the GPU, and each one's points, top-k and status equal tune_eval's bit for bit. A call whose queue of
descriptor groups another call uses or resets leaves points unwritten; a call whose status word another call
clears does not report its malformed descriptor. 20 threads are more than the 16 headers of the static array.

Marked run_last, as the other tests of this entry point."""

import threading

import pytest

from workloads import archs, gen

pytestmark = [pytest.mark.gpu, pytest.mark.run_last]


@pytest.mark.parametrize("threads", [2, 20])
def test_overlapping_calls(threads):
    import torch

    import paper_1701_08547_gb300 as T

    a, ax, k, n = archs.arch("sm_103"), gen.axes(), 5, 3000
    types = (torch.int32, torch.int32, torch.float32)
    jobs = []
    for i in range(threads):
        d = gen.descriptors(n, 50 + i, "uneven")
        if i % 3 == 2:  # this caller's descriptors hold a malformed one
            d["d"][n // 2] = 2.0
        off = gen.point_offsets(d)
        dd, po = T.descs_to_device(d), torch.from_numpy(off).cuda()
        ref = [torch.full((int(off[-1]),), 7, dtype=t, device="cuda") for t in types]
        top = T.tune_eval(a, ax, dd, k, flags=T.TUNE_EMIT_POINTS, pt_blocks=ref[0], pt_warps=ref[1], pt_cost=ref[2],
                          pt_offsets=po)
        jobs.append((dd, po, [*top, *ref], i % 3 == 2))
    torch.cuda.synchronize()
    start, failed = threading.Barrier(threads), []

    def run(dd, po, ref, malformed):
        stream = torch.cuda.Stream()
        with torch.cuda.stream(stream):
            got = [torch.empty_like(r) for r in ref]
        start.wait()
        for _ in range(6):
            with torch.cuda.stream(stream):
                for g in got:
                    g.fill_(7)
                try:
                    T.tune_eval_noalloc(a, ax, dd, k, flags=T.TUNE_EMIT_POINTS, topk_idx=got[0], topk_cost=got[1],
                                        pt_blocks=got[2], pt_warps=got[3], pt_cost=got[4], pt_offsets=po, stream=stream)
                    reported = False
                except T.TuneError:
                    reported = True
                same = [torch.equal(g.view(torch.int32), r.view(torch.int32)) for g, r in zip(got, ref)]
            if reported != malformed or not all(same):
                failed.append((reported, malformed, same))

    workers = [threading.Thread(target=run, args=j) for j in jobs]
    for w in workers:
        w.start()
    for w in workers:
        w.join()
    assert not failed, failed[:3]
