#!/usr/bin/env python
"""Benchmark of the PCR decode path: decoded images/s at scan group k on B200.

One step = one pcr_decode of one synthetic ImageNet-shaped record (1024 images, sizes
256..496, quality 90, 4:2:0, ten scans, restart every MCU row) at fidelity k: restart-interval
index, Huffman decode of scans 1..k into int16 coefficient lists and refinement side data, then blocks expanded and
refined, dequantise / inverse DCT / upsample / colour convert to packed RGB.  `value` is measured with the
record already resident in device memory; `e2e` copies the record prefix from pinned host
memory inside every step and reads the status words back.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--k 10] [--impl ours|reference]

With N > 1 (launched by torchrun, one rank per GPU) every rank decodes its own record of the
same distribution: independent units, no collective on the data path.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "decoded images/sec at scan group k"
UNIT = "images/s"
WORKLOAD = 1                 # ImageNet-shaped record
WORKLOAD_DESC = ("imagenet_shaped: 1 record x 1024 images per GPU, W,H in {256..496 step 16}, q90, 4:2:0, "
                 "10-scan script, restart per MCU row")
FALLBACK_HBM_GBS = 6650.0


# ----------------------------------------------------------------------------------------
# pieces shared by every rank (kept importable: the CPU tests exercise them over gloo)
# ----------------------------------------------------------------------------------------
def rank_record_index(rank: int) -> int:
    """Rank r decodes record r of the workload's distribution (weak scaling, no exchange)."""
    return rank


def _reduce(value: float, world_size: int, op_name: str) -> float:
    if world_size <= 1:
        return value
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([value], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=getattr(dist.ReduceOp, op_name))
    return float(t.item())


def reduce_max(value: float, world_size: int) -> float:
    """Max over ranks of a host-side scalar (the timed region)."""
    return _reduce(value, world_size, "MAX")


def reduce_sum(value: float, world_size: int) -> float:
    return _reduce(value, world_size, "SUM")


def whole_job_rate(images_this_rank: int, steps: int, ms_this_rank: float, world_size: int) -> float:
    """Images of all ranks / slowest rank's time."""
    total = reduce_sum(float(images_this_rank), world_size)
    ms = reduce_max(ms_this_rank, world_size)
    return total * steps / (ms / 1000.0)


def algorithmic_bytes(scans, infos, k: int, chains: bool = False):
    """Bytes of one decode at fidelity k through planes of whole blocks, per stage: a fixed measure of the work, reported as
    `plane_model_bytes_per_step` and nowhere else (this implementation keeps lists and moves layout_bytes).

    scans: [(ncomp, comp0, Ss, Se, Ah, wave, group_bytes)], infos: [(W, H)].
      index    : bytes of scan groups <= k, read once
      entropyW : compressed bytes of the wave's scans + 2 bytes per coefficient of every
                 block the scan visits (written once by a first pass, read and written by a
                 refinement)
      chains   : (records without restart markers) the AC refinements' share of the above, when the
                 library runs them as one stage of their own
      clear    : 128 bytes per block
      pixels   : 128 bytes per block read + 3 bytes per pixel written
    """
    out = {"index": 0.0, "clear": 0.0, "pixels": 0.0}
    ac_refine = {}
    blocks_pad = 0
    blocks_unp = [0, 0, 0]
    px = 0
    for W, H in infos:
        mx, my = (W + 15) // 16, (H + 15) // 16
        blocks_pad += 6 * mx * my
        cw, ch = (W + 1) // 2, (H + 1) // 2
        blocks_unp[0] += ((W + 7) // 8) * ((H + 7) // 8)
        blocks_unp[1] += ((cw + 7) // 8) * ((ch + 7) // 8)
        blocks_unp[2] += ((cw + 7) // 8) * ((ch + 7) // 8)
        px += W * H
    out["clear"] = 128.0 * blocks_pad
    out["pixels"] = 128.0 * blocks_pad + 3.0 * px
    for s, (ncomp, comp0, Ss, Se, Ah, wave, gbytes) in enumerate(scans):
        if s >= k:
            break
        out["index"] += gbytes
        band = Se - Ss + 1
        nb = blocks_pad if ncomp > 1 else blocks_unp[comp0]
        key = f"entropy{wave}"
        out[key] = out.get(key, 0.0) + gbytes + 2.0 * band * nb * (2 if Ah else 1)
        if Ah and Ss > 0:
            ac_refine[key] = ac_refine.get(key, 0.0) + gbytes + 4.0 * band * nb
    out["total"] = sum(out.values())
    if chains:          # the AC refinements ran as one stage of their own: their share moves there
        out["chains"] = 0.0
        for key, v in ac_refine.items():
            out[key] -= v
            out["chains"] += v
    return out


def layout_bytes(scans, infos, k: int, chains: bool = False):
    """Bytes the stages of one decode at fidelity k exchange with memory in the layout the library keeps (4:2:0), as far as
    they follow from the shapes: the non-zero values and the records of non-empty blocks that AC first passes write
    depend on the contents and are not counted, so this is a lower bound.  Arguments as for algorithmic_bytes.
      index    : bytes of scan groups <= k read, the copy without stuffing written
      entropyW : that copy read; a DC first pass writes 2 bytes per block, a DC refinement reads and writes them; an AC
                 refinement reads 8 bytes per block and mask source and writes 32 per block
      chains   : the AC refinements' share, when they ran as one stage of their own
      pixels   : per block 2 bytes DC and 16 of positions 1..7 (no AC scan: DC alone), 16 per first pass that reaches
                 beyond position 7, 32 per refinement; 3 bytes per pixel written
    """
    out = {"index": 0.0, "pixels": 0.0}
    pad, unp, px = [0, 0, 0], [0, 0, 0], 0
    for W, H in infos:
        mcus = ((W + 15) // 16) * ((H + 15) // 16)
        cw, ch = (W + 1) // 2, (H + 1) // 2
        for c, (n, w, h) in enumerate(((4 * mcus, W, H), (mcus, cw, ch), (mcus, cw, ch))):
            pad[c] += n
            unp[c] += ((w + 7) // 8) * ((h + 7) // 8)
        px += W * H
    chain_bytes = 0.0
    any_ac = any(Se > 0 for _, _, _, Se, _, _, _ in scans[:k])
    out["pixels"] = 3.0 * px + (18.0 if any_ac else 2.0) * sum(pad)
    for s, (ncomp, comp0, Ss, Se, Ah, wave, gbytes) in enumerate(scans[:k]):
        out["index"] += 2.0 * gbytes
        blocks = sum(pad) if ncomp > 1 else pad[comp0]
        moved = float(gbytes)
        if Ss == 0:
            moved += (4.0 if Ah else 2.0) * blocks
        elif Ah:
            before = [t for t in range(s) if scans[t][2] > 0 and scans[t][1] == comp0 and scans[t][2] <= Se and Ss <= scans[t][3]]
            sources = [t for t in before if not any(u > t and scans[u][4] and scans[u][2] <= scans[t][2] and scans[u][3] >= scans[t][3] for u in before)]
            moved += (32.0 + 8.0 * len(sources)) * unp[comp0]
        if Se >= 8 or Ah and Ss > 0:
            out["pixels"] += (32.0 if Ah else 16.0) * blocks
        if chains and Ah and Ss > 0:
            chain_bytes += moved
        else:
            out[f"entropy{wave}"] = out.get(f"entropy{wave}", 0.0) + moved
    if chains:
        out["chains"] = chain_bytes
    out["total"] = sum(out.values())
    return out


def source_code(text: str) -> str:
    """C++ source without comments, runs of white space as one space: what a compiler makes kernels of, whatever is written about them."""
    import re
    return re.sub(r'"(?:\\.|[^"\\\n])*"|((?:\s|//[^\n]*|/\*.*?\*/)+)', lambda m: " " if m.group(1) else m.group(0), text, flags=re.S)


def source_hash() -> str:
    """Hash of the CUDA sources (their code, not their comments): ncu counters are only quoted for the kernels they were taken on."""
    import glob
    import hashlib
    h = hashlib.sha256()
    for f in sorted(glob.glob(os.path.join(ROOT, "paper_1911_00472_b200", "csrc", "*"))):
        with open(f, encoding="utf-8") as fh:
            h.update(source_code(fh.read()).encode())
    return h.hexdigest()[:16]


def _traffic_table():
    """The committed ncu DRAM counters (profiles/traffic_imagenet_shaped.json), or None when the
    CUDA sources have changed since they were taken."""
    try:
        with open(os.path.join(ROOT, "profiles", "traffic_imagenet_shaped.json")) as f:
            t = json.load(f)
        return t if t["source_sha256_16"] == source_hash() else None
    except Exception:
        return None


def measured_traffic(stage: str, k: int, n_images: int):
    """dram__bytes_read + dram__bytes_write per launch of a stage's kernel (whole record in one
    launch) from the committed ncu capture at fidelity k, or None when the kernels changed since
    or the case was not captured."""
    t = _traffic_table()
    if t is None or n_images != 1024:
        return None
    return t["by_k"].get(str(k), {}).get("bytes_per_launch", {}).get(stage)


def measured_bytes_per_decode(k: int, n_images: int):
    """All DRAM bytes one decode at fidelity k moves (kernels' ncu counters plus the size of the
    status words' memset), from the committed capture, or None."""
    t = _traffic_table()
    if t is None or n_images != 1024:
        return None
    e = t["by_k"].get(str(k))
    if not e:
        return None
    return float(sum(e["bytes_per_launch"].values()) + e.get("memset_bytes", 0.0))


class ClockSampler:
    """SM clock and throttle-reason samples (NVML, read-only queries) taken by a thread while
    the timed region runs."""

    def __init__(self, gpu_index: int, period_s: float = 0.005):
        self.rows = []
        self.ok = False
        self._stop = threading.Event()
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            phys = gpu_index
            vis = os.environ.get("CUDA_VISIBLE_DEVICES")
            if vis:
                ids = [v.strip() for v in vis.split(",") if v.strip()]
                if gpu_index < len(ids) and ids[gpu_index].isdigit():
                    phys = int(ids[gpu_index])
            self.h = pynvml.nvmlDeviceGetHandleByIndex(phys)
            self.sm_max = float(pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM))
            self.period = period_s
            self.ok = True
            self.t = threading.Thread(target=self._run, daemon=True)
            self.t.start()
        except Exception as e:   # no NVML: report that, never guess
            self.err = repr(e)

    def _run(self):
        nv = self.nv
        while not self._stop.is_set():
            try:
                sm = float(nv.nvmlDeviceGetClockInfo(self.h, nv.NVML_CLOCK_SM))
                try:
                    rs = int(nv.nvmlDeviceGetCurrentClocksEventReasons(self.h))
                except Exception:
                    rs = int(nv.nvmlDeviceGetCurrentClocksThrottleReasons(self.h))
                try:
                    pw = nv.nvmlDeviceGetPowerUsage(self.h) / 1000.0
                except Exception:
                    pw = 0.0
                self.rows.append((time.perf_counter(), sm, rs, pw))
            except Exception:
                pass
            self._stop.wait(self.period)

    def stop(self, t0: float, t1: float):
        if not self.ok:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["NVML unavailable: " + getattr(self, "err", "")]}
        self._stop.set()
        self.t.join(timeout=2)
        rows = [r for r in self.rows if t0 <= r[0] <= t1]
        where = "timed region"
        if not rows:
            rows, where = self.rows, "whole run (timed region shorter than one sample)"
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": self.sm_max, "reasons": ["no samples"]}
        bits = {"hw_slowdown": 0x8, "hw_thermal_slowdown": 0x40, "sw_thermal_slowdown": 0x20, "sw_power_cap": 0x4}
        reasons = [n for n, b in bits.items() if any(r[2] & b for r in rows)]
        return {"sm_mhz": statistics.median(r[1] for r in rows), "sm_max_mhz": self.sm_max,
                "power_w_max": max(r[3] for r in rows), "samples": len(rows), "window": where, "reasons": reasons}


# ----------------------------------------------------------------------------------------
# CPU oracle timing (the reported baseline, and the --impl reference arm)
# ----------------------------------------------------------------------------------------
def _oracle_worker(args):
    path, k, lo, hi = args
    import numpy as np
    from oracle import pcr_oracle as O
    rec = np.load(path)
    for i in range(lo, hi):
        O.decode_image(rec, i, k, True)
    return hi - lo


def _oracle_crc_worker(args):
    """CRC-32 of the oracle's RGB bytes of images lo..hi-1 at fidelity k (the parity gate)."""
    path, k, lo, hi = args
    import zlib
    import numpy as np
    from oracle import pcr_oracle as O
    rec = np.load(path)
    return [(i, zlib.crc32(O.decode_image(rec, i, k, True)[1].tobytes())) for i in range(lo, hi)]


def oracle_crcs(pool, cores: int, rec_path: str, k: int, images) -> dict:
    """{image: CRC-32 of its oracle pixels at fidelity k} for a list of consecutive image indices."""
    lo0, hi0 = images[0], images[-1] + 1
    per = max(1, (hi0 - lo0 + cores * 2 - 1) // (cores * 2))
    shards = [(rec_path, k, lo, min(lo + per, hi0)) for lo in range(lo0, hi0, per)]
    out = {}
    for part in pool.map(_oracle_crc_worker, shards):
        out.update(part)
    return out


def device_crcs(dec, out, images) -> dict:
    """CRC-32 of the decoded pixels of the listed images (read back from the device)."""
    import zlib
    res = {}
    for i in images:
        inf = dec.info[i]
        res[i] = zlib.crc32(out[inf.out_offset:inf.out_offset + inf.out_bytes].cpu().numpy().tobytes())
    return res


def time_oracle(pool, cores: int, rec_path: str, k: int, n_images: int, passes: int = 1) -> float:
    """Images/s of the oracle decoding images [0, n_images) on `cores` processes."""
    per = max(1, (n_images + cores * 4 - 1) // (cores * 4))
    shards = [(rec_path, k, lo, min(lo + per, n_images)) for lo in range(0, n_images, per)]
    t0 = time.perf_counter()
    done = 0
    for _ in range(passes):
        done += sum(pool.map(_oracle_worker, shards))
    return done / (time.perf_counter() - t0)


def run_reference(args, rank: int):
    """The CPU oracle, as it stands, on this machine's host cores: same metric, config and unit."""
    if rank != 0:
        return
    import multiprocessing as mp
    import tempfile
    import numpy as np
    import pcr_synth
    from oracle import pcr_oracle as O
    O.build()
    cores = len(os.sched_getaffinity(0))
    rec = pcr_synth.make_record(WORKLOAD, 0)
    sample = min(rec.n_images, 256)
    with tempfile.TemporaryDirectory() as td:
        path = os.path.join(td, "rec.npy")
        np.save(path, rec.bytes)
        with mp.get_context("spawn").Pool(cores) as pool:
            for _ in range(max(args.warmup, 1)):
                time_oracle(pool, cores, path, args.k, min(sample, 64))
            t0 = time.perf_counter()
            for _ in range(args.steps):
                time_oracle(pool, cores, path, args.k, sample)
            dt = time.perf_counter() - t0
    value = sample * args.steps / dt
    desc = f"first {sample} images of the record per step, decoded by the single-threaded oracle in {cores} processes"
    print(json.dumps({
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1000.0 * dt / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "int16/u8", "data": "synthetic",
        "config": {"workload": WORKLOAD_DESC, "k": args.k},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": desc},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }))


def streamed_sweep(dev, recs, ks, peak, pool=None, cores=0, tmpdir=None):
    """Throughput sweep (the fifth workload): R ImageNet-shaped records of 1024 images, streamed
    from pinned host memory on two CUDA streams (two records in flight: the copy of one overlaps
    the decode of the other), every record opened, copied, decoded and closed once per k.

    Parity: before the timed passes of a k every record goes through the same streamed path once
    and the CRC-32 of every image's pixels is compared with the oracle's (when the oracle pool of
    the CPU baseline is available); after the timed pass the outputs of the last two records are
    compared on the device with a resident decode of the same records."""
    import zlib
    from concurrent.futures import ThreadPoolExecutor
    import numpy as np
    import torch
    from paper_1911_00472_b200 import Decoder, binding
    R = len(recs)
    decs = [Decoder(r.bytes, device=dev) for r in recs]
    n_img = sum(d.n_images for d in decs)
    streams = [torch.cuda.Stream(dev), torch.cuda.Stream(dev)]
    size = max(d.out_bytes for d in decs)
    outs = [torch.zeros(size, dtype=torch.uint8, device=dev) for _ in range(2)]
    check = torch.zeros(size, dtype=torch.uint8, device=dev)
    scans0 = []
    for s in range(decs[0].n_groups):
        si = binding.pcr_get_scan(decs[0].handle, s)
        scans0.append((si.ncomp, si.comp[0], si.Ss, si.Se, si.Ah, si.wave))
    per_k = {}
    OPEN_AHEAD = 3
    opener = ThreadPoolExecutor(max_workers=OPEN_AHEAD, initializer=lambda: torch.cuda.set_device(dev))
    hasher = ThreadPoolExecutor(max_workers=8)
    rec_paths = []
    if pool is not None:
        for r, rec in enumerate(recs):
            path = os.path.join(tmpdir, f"sweep_rec{r}.npy")
            np.save(path, rec.bytes)
            rec_paths.append(path)

    def image_crcs(d, host):
        def one(i):
            inf = d.info[i]
            return zlib.crc32(host[inf.out_offset:inf.out_offset + inf.out_bytes])
        return list(hasher.map(one, range(d.n_images)))

    for k in ks:
        # ---- parity of the streamed path against the oracle, every image of every record
        checked = 0
        if pool is not None:
            for i, d in enumerate(decs):
                want = oracle_crcs(pool, cores, rec_paths[i], k, list(range(d.n_images)))
                h = binding.pcr_open(d.host.data_ptr(), d.host.numel())
                binding.pcr_decode(h, k, outs[i & 1].data_ptr(), streams[i & 1].cuda_stream)
                streams[i & 1].synchronize()
                bad, code = binding.pcr_status(h)
                binding.pcr_close(h)
                if code != 0:
                    raise RuntimeError(f"sweep: decode error {code} on image {bad} of record {i}")
                got = image_crcs(d, memoryview(outs[i & 1].cpu().numpy()))
                for j in range(d.n_images):
                    if got[j] != want[j]:
                        raise RuntimeError(f"sweep parity: record {i} image {j} differs from the oracle at k={k}")
                checked += d.n_images
        rates = {}
        for rep in range(4):
            # passes 0, 1: every open parses the record (pass 0 warms up, pass 1 is timed); passes 2, 3: with
            # the cache of closed records on, as in the second and later epochs of a loader (pass 2 fills it)
            if rep == 2:
                binding.pcr_set_record_cache(64 << 30)
            torch.cuda.synchronize(dev)
            t0 = time.perf_counter()
            live = []                            # handles of the records in flight, at most two
            # every record is opened, copied and decoded once, as a loader streaming a data set does.
            # Loader threads parse the next records (pcr_open: host-side marker walk and table
            # uploads) while this thread enqueues decodes.
            ahead = [opener.submit(binding.pcr_open, d.host.data_ptr(), d.host.numel()) for d in decs[:OPEN_AHEAD]]
            last = []
            for i, d in enumerate(decs):
                h = ahead.pop(0).result()
                if i + OPEN_AHEAD < len(decs):
                    nd = decs[i + OPEN_AHEAD]
                    ahead.append(opener.submit(binding.pcr_open, nd.host.data_ptr(), nd.host.numel()))
                binding.pcr_decode(h, k, outs[i & 1].data_ptr(), streams[i & 1].cuda_stream)
                live.append(h)
                if len(live) > 2:
                    old = live.pop(0)
                    binding.pcr_close(old)       # waits for that record's decode only
            torch.cuda.synchronize(dev)
            dt = time.perf_counter() - t0
            for h in live:
                bad, code = binding.pcr_status(h)
                if code != 0:
                    raise RuntimeError(f"sweep: decode error {code} on image {bad}")
                binding.pcr_close(h)
            rates[rep] = dt
        binding.pcr_set_record_cache(0)
        dt = rates[1]
        # the outputs the timed pass left behind (last two records) against a resident decode
        for i in range(max(0, R - 2), R):
            d = decs[i]
            d.decode(k, check)
            torch.cuda.synchronize(dev)
            bad, code = d.status()
            if code != 0:
                raise RuntimeError(f"decode error {code} on image {bad}")
            for inf in d.info:
                a, b = inf.out_offset, inf.out_offset + inf.out_bytes
                if not torch.equal(outs[i & 1][a:b], check[a:b]):
                    raise RuntimeError(f"sweep: streamed output of record {i} differs from the resident decode at k={k}")
        model = 0.0
        h2d = 0
        for d in decs:
            scans = [sc + (binding.pcr_get_scan(d.handle, s).bytes,) for s, sc in enumerate(scans0)]
            model += layout_bytes(scans, [(i.width, i.height) for i in d.info], k)["total"]
            h2d += d.prefix_bytes(k)
        per_k[str(k)] = {"images_per_s": n_img / dt, "ms_per_record": 1000.0 * dt / R, "hbm_gbs_model": model / dt / 1e9,
                         "model_frac_of_peak": model / dt / 1e9 / peak, "h2d_bytes_per_record": h2d // R,
                         "images_per_s_records_seen_before": n_img / rates[3],
                         "parity_images_vs_oracle": checked}
    n_per = decs[0].n_images
    for d in decs:
        d.close()
    opener.shutdown()
    hasher.shutdown()
    return {"workload": f"sweep: {R} ImageNet-shaped records x {n_per} images, streamed from pinned host memory on two CUDA "
                        "streams, each record opened (host parse, three loader threads ahead), copied, decoded and closed once per k, two in flight",
            "timing": "wall clock around enqueue + synchronise, second of two passes; images_per_s_records_seen_before: the same "
                      "with pcr_set_record_cache on, every record having been opened and closed once before (a later epoch)",
            "parity": "every image of every record against the oracle's CRC-32 (streamed path, before timing) when the oracle pool runs; "
                      "the last two streamed outputs against a resident decode on the device",
            "by_k": per_k}


def hbm_peak():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return float(json.load(f)["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


def run_sweep(args):
    """The full sweep on its own: --records records, k = 1..10."""
    import multiprocessing as mp
    import tempfile
    import pcr_synth
    pool, cores, tmp = None, len(os.sched_getaffinity(0)), tempfile.TemporaryDirectory()
    if not args.no_cpu_baseline:
        from oracle import pcr_oracle as O
        O.build()
        pool = mp.get_context("spawn").Pool(cores)
        pool.map(abs, range(cores))              # start the workers before the first GPU call
    import torch
    from paper_1911_00472_b200 import build as libbuild
    libbuild.build()
    dev = torch.device("cuda", 0)
    torch.cuda.set_device(dev)
    recs = [pcr_synth.make_record(4, r, n_images=args.images or None) for r in range(args.records)]
    res = streamed_sweep(dev, recs, list(range(1, 11)), hbm_peak()[0], pool, cores, tmp.name)
    print(json.dumps({"metric": METRIC, "unit": UNIT, "n_gpus": 1, "data": "synthetic", "dtype": "int16/u8",
                      "config": {"workload": res["workload"], "timing": res["timing"], "parity": res["parity"]},
                      "sweep": res["by_k"]}))
    if pool is not None:
        pool.close(); pool.join()
    tmp.cleanup()


# ----------------------------------------------------------------------------------------
def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--k", type=int, default=10, help="scan group (fidelity) of the headline number")
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", type=int, default=WORKLOAD, choices=[1, 2, 3],
                    help="1 ImageNet-shaped (the headline), 2 CelebA-shaped, 3 HAM10000-shaped (no restart markers)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--headline-only", action="store_true",
                    help="only the timed steps, the end-to-end loop and the stage profile (no per-k, tensor, fidelity extras)")
    ap.add_argument("--images", type=int, default=0, help="images per record (default: the workload's 1024)")
    ap.add_argument("--sweep", action="store_true", help="run the streamed multi-record sweep over k = 1..10 instead")
    ap.add_argument("--records", type=int, default=16, help="records of the sweep")
    args = ap.parse_args()

    rank = int(os.environ.get("RANK", "0"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    if args.impl == "reference":
        run_reference(args, rank)
        return
    if args.sweep:
        if rank == 0:
            run_sweep(args)
        return
    args.warmup = max(args.warmup, 3)

    import multiprocessing as mp
    import tempfile
    import numpy as np
    import pcr_synth

    # input record of this rank; the oracle's process pool starts before the first GPU call
    wl = args.workload
    wl_desc = WORKLOAD_DESC if wl == WORKLOAD else {
        2: "celeba_shaped: 1 record x 1024 images per GPU, 178x218, q95, 4:2:0, 10-scan script, restart per MCU row",
        3: "ham10000_shaped: 1 record x 1024 images per GPU, 600x450, q90, 4:2:0, 10-scan script, no restart markers"}[wl]
    rec = pcr_synth.make_record(wl, rank_record_index(rank), n_images=args.images or None)
    pool = None
    tmpdir = None
    cores = len(os.sched_getaffinity(0))
    do_cpu = (rank == 0 and world == 1 and not args.no_cpu_baseline)
    if do_cpu:
        from oracle import pcr_oracle as O
        O.build()
        tmpdir = tempfile.TemporaryDirectory()
        rec_path = os.path.join(tmpdir.name, "rec.npy")
        np.save(rec_path, rec.bytes)
        pool = mp.get_context("spawn").Pool(cores)
        time_oracle(pool, cores, rec_path, 1, min(64, rec.n_images))   # start the workers
        # parity gate: the oracle's pixels of a sample of the timed record at the timed fidelity
        # (CRC-32 per image), compared with the device output before anything is timed
        parity_images = list(range(min(rec.n_images, 128)))
        parity_want = oracle_crcs(pool, cores, rec_path, args.k, parity_images)
    sweep_recs = []
    if do_cpu and wl == WORKLOAD and not args.headline_only and not args.images:
        sweep_recs = [pcr_synth.make_record(4, r) for r in range(4)]

    import torch
    import torch.distributed as dist
    from paper_1911_00472_b200 import Decoder, binding
    from paper_1911_00472_b200 import build as libbuild
    libbuild.build()
    torch.cuda.set_device(local_rank)
    dev = torch.device("cuda", local_rank)
    if world > 1:
        dist.init_process_group("nccl", device_id=dev)
    dec = Decoder(rec.bytes, device=dev)
    out = dec.alloc_out()
    stream = torch.cuda.current_stream(dev)
    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)     # > 126 MB L2
    k = args.k
    n_img = dec.n_images
    scans = []
    for s in range(dec.n_groups):
        si = binding.pcr_get_scan(dec.handle, s)
        scans.append((si.ncomp, si.comp[0], si.Ss, si.Se, si.Ah, si.wave, si.bytes))
    infos = [(i.width, i.height) for i in dec.info]

    def sync_all():
        torch.cuda.synchronize(dev)
        if world > 1:
            dist.barrier()
            torch.cuda.synchronize(dev)

    def timed_steps(kk, steps):
        """Sum of per-step device times (ms): L2 flushed before every step, events on the launch stream."""
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        for a, b in evs:
            flush.fill_(1)
            a.record(stream)
            dec.decode(kk, out)
            b.record(stream)
        torch.cuda.synchronize(dev)
        return sum(a.elapsed_time(b) for a, b in evs)

    dec.decode(k, out)
    torch.cuda.synchronize(dev)
    bad, code = dec.status()
    if code != 0:
        raise RuntimeError(f"decode reported error {code} on image {bad}")
    parity_checked = None
    if do_cpu:
        got = device_crcs(dec, out, parity_images)
        diff = [i for i in parity_images if got[i] != parity_want[i]]
        if diff:
            raise RuntimeError(f"parity: images {diff[:8]} differ from the oracle at k={k}")
        parity_checked = {"images": len(parity_images), "k": k, "how": "CRC-32 of every sampled image's RGB bytes, device output "
                          "against the CPU oracle, before the timed steps"}

    sampler = ClockSampler(local_rank)
    for _ in range(args.warmup):
        dec.decode(k, out)
    sync_all()
    launches0 = binding.pcr_launch_count()
    t0 = time.perf_counter()
    ms = timed_steps(k, args.steps)
    t1 = time.perf_counter()
    launches = binding.pcr_launch_count() - launches0
    sync_all()
    clocks = sampler.stop(t0, t1)
    ms_max = reduce_max(ms, world)
    total_images = reduce_sum(float(n_img), world)
    value = total_images * args.steps / (ms_max / 1000.0)

    # end to end: prefix copied from pinned host memory inside every step, status words read back
    prefix = dec.prefix_bytes(k)
    for _ in range(2):
        dec.evict(); dec.decode(k, out); torch.cuda.synchronize(dev); dec.status()
    sync_all()
    te = time.perf_counter()
    for _ in range(args.steps):
        dec.evict()
        dec.decode(k, out)
        torch.cuda.synchronize(dev)
        dec.status()
    e2e_s = reduce_max(time.perf_counter() - te, world)
    e2e = {"value": total_images * args.steps / e2e_s, "unit": UNIT, "h2d_bytes_per_step": int(prefix),
           "d2h_bytes_per_step": 4 * n_img, "ms_per_step": 1000.0 * e2e_s / args.steps,
           "note": "pcr_evict + pcr_decode from pinned host bytes + synchronise + pcr_status, wall clock; "
                   "pixels stay on the device for the training step"}

    # the same with the record opened and closed inside every step (what a loader pays that sees
    # every record once: host-side parse, table uploads, copy, decode)
    n_open = max(5, min(args.steps, 30))

    def open_decode_close():
        h = binding.pcr_open(dec.host.data_ptr(), dec.host.numel())
        binding.pcr_decode(h, k, out.data_ptr(), stream.cuda_stream)
        torch.cuda.synchronize(dev)
        binding.pcr_status(h)
        binding.pcr_close(h)

    for _ in range(2):                 # the first opens allocate the second record's device buffers
        open_decode_close()
    sync_all()
    to = time.perf_counter()
    for _ in range(n_open):
        open_decode_close()
    open_s = reduce_max(time.perf_counter() - to, world)
    e2e["with_open_close"] = {"value": total_images * n_open / open_s, "unit": UNIT, "ms_per_step": 1000.0 * open_s / n_open,
                              "note": "pcr_open + pcr_decode from pinned host bytes + synchronise + pcr_status + pcr_close per step"}
    binding.pcr_set_record_cache(8 << 30)
    for _ in range(2):
        open_decode_close()
    sync_all()
    to = time.perf_counter()
    for _ in range(n_open):
        open_decode_close()
    open_s = reduce_max(time.perf_counter() - to, world)
    binding.pcr_set_record_cache(0)
    e2e["with_open_close_record_seen_before"] = {
        "value": total_images * n_open / open_s, "unit": UNIT, "ms_per_step": 1000.0 * open_s / n_open,
        "note": "the same with pcr_set_record_cache on: the record was opened and closed before, as in a loader's later epochs"}

    per_k, raise_ms, training_tensor, fidelity, baseline_jpeg = {}, {}, None, None, None
    hbm_by_k, hbm_meas_by_k = {}, {}
    triangle = None
    sweep = None
    if not args.headline_only:
        # per-k numbers and the stage profile (this rank's GPU)
        per_k = {}
        for kk in pcr_synth.WORKLOADS[wl].ks:
            for _ in range(2):
                dec.decode(kk, out)
            torch.cuda.synchronize(dev)
            st = 5
            per_k[str(kk)] = n_img * st / (timed_steps(kk, st) / 1000.0)
            hbm_by_k[str(kk)] = layout_bytes(scans, infos, kk)["total"] * per_k[str(kk)] / n_img / 1e9
            mb = measured_bytes_per_decode(kk, n_img) if wl == WORKLOAD else None
            hbm_meas_by_k[str(kk)] = mb * per_k[str(kk)] / n_img / 1e9 if mb is not None else None
        # decode straight to a fixed-size training batch (random-resized crops, flip, 224 x 224, fp16)
        crops = pcr_synth.random_resized_crops(infos, 1000 + rank)
        t_size = 224
        t_mean, t_std = (0.485, 0.456, 0.406), (0.229, 0.224, 0.225)
        tensor = torch.empty((n_img, 3, t_size, t_size), dtype=torch.float16, device=dev)
        tensor_by_k = {}
        for kk in pcr_synth.WORKLOADS[wl].ks:
            for _ in range(2):
                dec.decode_tensor(kk, crops, t_size, t_mean, t_std, rgb=out, tensor=tensor)
            torch.cuda.synchronize(dev)
            st, acc = 5, 0.0
            for _ in range(st):
                flush.fill_(1)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                dec.decode_tensor(kk, crops, t_size, t_mean, t_std, rgb=out, tensor=tensor)
                b.record(stream)
                torch.cuda.synchronize(dev)
                acc += a.elapsed_time(b)
            tensor_by_k[str(kk)] = n_img * st / (acc / 1000.0)
        crop_frac = float(sum(int(c[2]) * int(c[3]) for c in crops)) / float(sum(w * h for w, h in infos))
        training_tensor = {"size": t_size, "dtype": "f16", "images_per_s_by_k": tensor_by_k,
                           "crop_area_fraction": crop_frac,
                           "note": "pcr_decode_tensor: random-resized crops (area 8-100 %, aspect 3/4-4/3), flip, bilinear, normalise; "
                                   "only the MCUs a crop touches are transformed"}
        # the paper's fidelity diagnostic: multi-scale SSIM of scan group k against full fidelity
        full = dec.alloc_out()
        dec.decode(dec.n_groups, full)
        ms_by_k = {}
        for kk in range(1, dec.n_groups):
            dec.decode(kk, out)
            sc = dec.msssim(out, full)
            torch.cuda.synchronize(dev)
            v = sc.float().cpu().numpy()
            ms_by_k[str(kk)] = {"mean": float(np.nanmean(v)), "q25": float(np.nanpercentile(v, 25)), "q75": float(np.nanpercentile(v, 75))}
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        for _ in range(5):
            dec.msssim(out, full)
        b.record(stream)
        torch.cuda.synchronize(dev)
        fidelity = {"msssim_vs_full_by_k": ms_by_k, "msssim_images_per_s": n_img * 5 / (a.elapsed_time(b) / 1000.0),
                    "note": "pcr_msssim on the decoded pixels of this record; the paper reports 95 %+ from scan group 5 on for its datasets"}
        del full
        # the comparison column of the paper's Table 2: the same images as baseline (sequential) JPEGs
        with pcr_synth.scan_script(pcr_synth.SCRIPT_BASELINE):
            rec_b = pcr_synth.make_record(wl, rank_record_index(rank), n_images=args.images or None)
        dec_b = Decoder(rec_b.bytes, device=dev)
        for _ in range(3):
            dec_b.decode(1, out)
        torch.cuda.synchronize(dev)
        if dec_b.status()[1] != 0:
            raise RuntimeError("baseline record: decode error")
        acc, st = 0.0, 10
        for _ in range(st):
            flush.fill_(1)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(stream)
            dec_b.decode(1, out)
            b.record(stream)
            torch.cuda.synchronize(dev)
            acc += a.elapsed_time(b)
        baseline_jpeg = {"images_per_s": n_img * st / (acc / 1000.0), "bytes_per_image": dec_b.prefix_bytes(1) / n_img,
                         "progressive_bytes_per_image": dec.prefix_bytes(dec.n_groups) / n_img,
                         "note": "a record of baseline JPEGs of the same images (one scan group), decoded by the same library; "
                                 "the paper's Table 2 has all ten progressive scans at less than half its baseline rate on a CPU"}
        dec_b.close()
        del rec_b
        # triangle chroma upsampling (the stock decoders' filter) instead of 2x2 replication
        dec.set_upsampling(True)
        for _ in range(2):
            dec.decode(k, out)
        torch.cuda.synchronize(dev)
        triangle = {"k": k, "images_per_s": n_img * 5 / (timed_steps(k, 5) / 1000.0)}
        dec.set_upsampling(False)
        # raising the fidelity of a resident decode: only the new scan groups are decoded
        raise_ms = {}
        for k_from, k_to in ((1, 10), (5, 10), (2, 5)):
            if k_to > dec.n_groups:
                continue
            acc = 0.0
            reps = 5
            for _ in range(reps):
                dec.decode(k_from, out)
                flush.fill_(1)
                a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                a.record(stream)
                dec.decode_more(k_to, out)
                b.record(stream)
                torch.cuda.synchronize(dev)
                acc += a.elapsed_time(b) / reps
            raise_ms[f"{k_from}->{k_to}"] = acc
    if sweep_recs:
        # the streamed multi-record workload, short form: 4 records, k = 1, 5, 10
        sweep = streamed_sweep(dev, sweep_recs, [1, 5, 10], hbm_peak()[0], pool, cores, tmpdir.name)
        del sweep_recs
    binding.pcr_set_profiling(dec.handle, True)
    stage_ms, stage_n = {}, {}
    reps = 5
    for _ in range(reps):
        flush.fill_(1)
        dec.decode(k, out)
        torch.cuda.synchronize(dev)
        for name, t, nl in binding.pcr_get_profile(dec.handle):
            stage_ms[name] = stage_ms.get(name, 0.0) + t / reps
            stage_n[name] = nl
    binding.pcr_set_profiling(dec.handle, False)
    model = layout_bytes(scans, infos, k, chains=stage_n.get("chains", 0) > 0)
    kernels = {n: t for n, t in stage_ms.items() if stage_n.get(n, 0) > 0}
    dom = max(kernels, key=kernels.get)
    peak, peak_src = hbm_peak()
    achieved = model[dom] / (kernels[dom] * 1e-3) / 1e9
    traffic = measured_traffic(dom, k, n_img) if wl == WORKLOAD else None      # the capture is of the ImageNet-shaped record
    whole = model["total"] / (ms_max / args.steps * 1e-3) / 1e9
    roofline = {"bound": "hbm", "kernel": dom, "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
                "traffic": traffic, "peak_source": peak_src, "kernel_ms": kernels[dom],
                "algorithmic_bytes_per_launch": model[dom],
                "whole_path": {"algorithmic_bytes_per_step": model["total"], "achieved": whole, "frac": whole / peak},
                "plane_model_bytes_per_step": algorithmic_bytes(scans, infos, k)["total"],
                "step_ms": {"pipelined": ms_max / args.steps, "stages_one_after_the_other": sum(stage_ms.values()),
                            "note": "value is timed in the pipelined layout (image slices on their own streams); the stage "
                                    "times below come from the profiling layout, one stage after the other"},
                "stages_ms": stage_ms,
                "stage_frac_of_peak": {n: (model.get(n, 0.0) / (t * 1e-3) / 1e9 / peak if t > 0 else None)
                                       for n, t in stage_ms.items()}}

    cpu_baseline = None
    if do_cpu:
        n_s = min(n_img, 512)
        v0 = time_oracle(pool, cores, rec_path, k, n_s, passes=1)
        passes = max(2, min(200, int(12.0 * v0 / n_s)))          # about 12 s of wall time on all cores
        v = time_oracle(pool, cores, rec_path, k, n_s, passes=passes)
        t1c = time.perf_counter()
        n1 = sum(pool.map(_oracle_worker, [(rec_path, k, 0, min(n_img, 48))]))      # one shard = one process
        v1 = n1 / (time.perf_counter() - t1c)
        pool.close(); pool.join()
        cpu_baseline = {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
                        "sample": f"images 0..{n_s - 1} of the same record at k={k}, {passes} passes, {cores} processes of the single-threaded oracle",
                        "one_core": v1}
        tmpdir.cleanup()

    # Theorem 1 of the paper: a data-bound pipeline speeds up by the ratio of mean sample sizes;
    # here full-fidelity bytes over the bytes of the record prefix that fidelity k reads
    io_speedup = {str(kk): dec.prefix_bytes(dec.n_groups) / dec.prefix_bytes(kk) for kk in range(1, dec.n_groups + 1)}
    if rank == 0:
        comp = [s[6] for s in scans]
        print(json.dumps({
            "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": ms_max / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "int16/u8", "data": "synthetic",
            "config": {"workload": wl_desc, "k": k, "images_per_step_per_gpu": n_img,
                       "l2": "flushed by a 256 MiB write before every timed step",
                       "record_bytes": int(rec.bytes.size), "prefix_bytes_at_k": int(prefix),
                       "mean_compressed_bytes_per_image_by_scan": [c / n_img for c in comp]},
            "e2e": e2e, "gpu_launches": int(launches), "clocks": clocks, "roofline": roofline,
            "cpu_baseline": cpu_baseline, "parity_checked": parity_checked, "sweep": sweep,
            "images_per_s_by_k": per_k, "hbm_gbs_model_by_k": hbm_by_k,
            "hbm_model_frac_of_peak_by_k": {kk: v / peak for kk, v in hbm_by_k.items()},
            "hbm_gbs_measured_by_k": hbm_meas_by_k,
            "hbm_measured_frac_of_peak_by_k": {kk: (v / peak if v is not None else None) for kk, v in hbm_meas_by_k.items()},
            "hbm_by_k_note": "model: bytes the stages of a decode at k exchange with memory in the library's layout, as far as they follow "
                             "from the shapes (compressed prefix read and copied without stuffing, DC and head planes, block records, "
                             "refinement side data, pixels; without the values of AC first passes) / time; part of it stays in L2.  "
                             "measured: DRAM bytes the kernels and memsets of one decode really move (ncu dram__bytes of every kernel, "
                             "committed under profiles/) / the same time; null when the kernels changed since the capture",
            "raise_fidelity_ms_per_record": raise_ms,
            "training_tensor": training_tensor, "predicted_io_speedup_by_k": io_speedup, "fidelity": fidelity, "baseline_jpeg": baseline_jpeg, "triangle_upsampling": triangle,
        }))
    dec.close()
    if world > 1:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
