"""The batch kernel against the general kernel of laq_gemm_wxg128, each in its planned shape.

    python -m paper_2605_08755_gb300.measure.kernel_choice --chain            # sizes x M x bits
    python -m paper_2605_08755_gb300.measure.kernel_choice --decoder 4096,6144,4096,12288
    python -m paper_2605_08755_gb300.measure.kernel_choice --shapes --K 4096 --N 1024

Two settings.  ``--chain``: a CUDA graph of dependent launches of one size (K, N) over as many
copies of a weight as exceed L2 (at most 24), for a grid of sizes.  ``--decoder H,QKV,O,I``: a graph
of whole layers (H x QKV, O x H, H x 2 I, I x H): every launch on the general kernel, as planned, and
for each projection it alone on the batch kernel (``alone``) and the plan with its kernel changed
(``changed``; launches of the two kernels overlap less than launches of one, so that the two
differ).  One JSON line per size, M and width: microseconds per call (chain) or per layer (decoder)
and whether laq_gemm_plan takes the batch kernel.  Where it does not, the batch kernel runs in the
shape planned for M = 5.  ``--shapes`` times every shape of the batch kernel (tiles per warp, tile
slots, cluster) in the chain, for the plan's choice among them.
"""
import argparse
import json

import torch

from .. import _lib
from ..weight_pass import QuantLinear

DEV = "cuda"


class Copy:
    def __init__(self, q):
        self.packed, self.s, self.z = q.packed.clone(), q.s.clone(), q.z.clone()


def configs(M, K, N, bits, sms):
    """(general, batch, planned on the batch kernel)"""
    plan = _lib.laq_gemm_plan(M, K, N, bits, sms)
    d = dict(plan.as_dict(), pdl=1)
    batch = d.pop("batch", None)
    forced = batch or _lib.laq_gemm_plan(max(M, 5), K, N, bits, sms).batch
    make = _lib.GemmConfig.make
    return make(**d), make(**d, batch=forced), batch is not None


def timed(launch, stream, calls):
    launch(None)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        launch(stream)
    best = float("inf")
    for _ in range(4):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        with torch.cuda.stream(stream):
            g.replay()
            a.record(stream)
            for _ in range(6):
                g.replay()
            b.record(stream)
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3 / 6 / calls)
    return best


def call(X, q, bits, Y, cfg, stream):
    _lib.laq_gemm_wxg128(X, q.packed, q.s, q.z, bits, Y=Y, config=cfg, stream=stream)


def weight(K, N, bits):
    return QuantLinear((torch.randn((K, N), device=DEV) * 0.02).half(), bits)


def chain(Ks, Ns, Ms, widths, sms, stream):
    for bits in widths:
        for K in Ks:
            for N in Ns:
                if K * N > 5e8:
                    continue
                q = weight(K, N, bits)
                n = max(1, min(24, int(3e8 // q.packed.numel())))
                qs = [q] + [Copy(q) for _ in range(n - 1)]
                reps = max(1, 24 // n)
                for M in Ms:
                    X = torch.randn((M, K), device=DEV).half()
                    Y = torch.empty((M, N), device=DEV, dtype=torch.float16)
                    general, batch, planned = configs(M, K, N, bits, sms)
                    t = [timed(lambda s: [call(X, w, bits, Y, cfg, s) for _ in range(reps)
                                          for w in qs], stream, n * reps)
                         for cfg in (general, batch)]
                    print(json.dumps(dict(bits=bits, K=K, N=N, M=M, general=round(t[0], 3),
                                          batch=round(t[1], 3), planned=planned,
                                          shape=batch.batch)), flush=True)


def shapes(Ks, Ns, Ms, widths, sms, stream):
    for bits in widths:
        for K in Ks:
            for N in Ns:
                q = weight(K, N, bits)
                n = max(1, min(24, int(3e8 // q.packed.numel())))
                qs = [q] + [Copy(q) for _ in range(n - 1)]
                reps = max(1, 24 // n)
                for M in Ms:
                    X = torch.randn((M, K), device=DEV).half()
                    Y = torch.empty((M, N), device=DEV, dtype=torch.float16)
                    general, batch, planned = configs(M, K, N, bits, sms)
                    run = lambda cfg: timed(lambda s: [call(X, w, bits, Y, cfg, s)
                                                       for _ in range(reps) for w in qs],
                                            stream, n * reps)
                    base = {k: v for k, v in general.as_dict().items() if k != "batch"}
                    t = {}
                    for tw in (1, 2):
                        for slots in (1, 2, 4, 8):
                            for cl in range(1, min(8, K // 128) + 1):
                                if -(-(N // 16) // (tw * slots)) * cl > 8 * sms:
                                    continue
                                c = _lib.GemmConfig.make(**base, batch=(tw, slots, cl))
                                t[f"{tw},{slots},{cl}"] = round(run(c), 3)
                    print(json.dumps(dict(bits=bits, K=K, N=N, M=M, general=round(run(general), 3),
                                          planned=planned, shape=batch.batch, batch=t)),
                          flush=True)


def decoder(dims, Ms, widths, sms, stream):
    H, QKV, O, I = dims
    sizes = [(H, QKV), (O, H), (H, 2 * I), (I, H)]
    for bits in widths:
        layer = [weight(K, N, bits) for K, N in sizes]
        n = max(2, min(24, int(4e8 // sum(q.packed.numel() for q in layer))))
        layers = [layer] + [[Copy(q) for q in layer] for _ in range(n - 1)]
        for M in Ms:
            X = [torch.randn((M, K), device=DEV).half() for K, _ in sizes]
            Y = [torch.empty((M, N), device=DEV, dtype=torch.float16) for _, N in sizes]
            cf = [configs(M, K, N, bits, sms) for K, N in sizes]

            def per_layer(on):
                def launch(s):
                    for qs in layers:
                        for j in range(4):
                            call(X[j], qs[j], bits, Y[j], cf[j][j in on], s)
                return timed(launch, stream, n)
            base = per_layer(())
            plan = [j for j in range(4) if cf[j][2]]
            line = dict(dims=dims, bits=bits, M=M, general=round(base, 2),
                        plan=round(per_layer(plan), 2))
            for j, name in enumerate(("qkv", "o", "gate_up", "down")):
                line[name] = dict(alone=round(per_layer((j,)), 2),
                                  changed=round(per_layer(sorted({j} ^ set(plan))), 2),
                                  planned=cf[j][2], shape=cf[j][1].batch)
            print(json.dumps(line), flush=True)


def main():
    ints = lambda s: [int(v) for v in s.split(",")]
    ap = argparse.ArgumentParser()
    ap.add_argument("--chain", action="store_true")
    ap.add_argument("--shapes", action="store_true")
    ap.add_argument("--decoder", type=ints, action="append", default=[], metavar="H,QKV,O,I")
    ap.add_argument("--K", type=ints, default=[128, 256, 512, 1024, 1408, 2048, 2560, 4096, 5120,
                                               8192, 12288])
    ap.add_argument("--N", type=ints, default=[16 * t for t in (
        1, 4, 16, 40, 64, 96, 128, 160, 256, 384, 512, 768, 1024, 1536, 2048, 4096, 9496)])
    ap.add_argument("--M", type=ints, default=[1, 2, 3, 4, 5, 8, 9, 16])
    ap.add_argument("--bits", type=ints, default=[3, 4])
    a = ap.parse_args()
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    stream = torch.cuda.Stream()
    if a.chain:
        chain(a.K, a.N, a.M, a.bits, sms, stream)
    if a.shapes:
        shapes(a.K, a.N, a.M, a.bits, sms, stream)
    for dims in a.decoder:
        decoder(dims, a.M, a.bits, sms, stream)


if __name__ == "__main__":
    main()
