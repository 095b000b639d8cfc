/* A stream of a green context: a stream limited to some of the GPU's SMs, for
 * the test of contexts on such streams.  Returns a CUresult. */
#include <cuda.h>

int green_stream(int device, unsigned int sms, CUgreenCtx *ctx, CUstream *stream)
{
    CUdevice dev;
    CUdevResource all, part;
    CUdevResourceDesc desc;
    unsigned int groups = 1;
    CUresult e = cuInit(0);
    if (!e) e = cuDeviceGet(&dev, device);
    if (!e) e = cuDeviceGetDevResource(dev, &all, CU_DEV_RESOURCE_TYPE_SM);
    if (!e) e = cuDevSmResourceSplitByCount(&part, &groups, &all, 0, 0, sms);
    if (!e) e = cuDevResourceGenerateDesc(&desc, &part, 1);
    if (!e) e = cuGreenCtxCreate(ctx, desc, dev, CU_GREEN_CTX_DEFAULT_STREAM);
    if (!e) e = cuGreenCtxStreamCreate(stream, *ctx, CU_STREAM_NON_BLOCKING, 0);
    return (int)e;
}

int green_free(CUgreenCtx ctx, CUstream stream)
{
    CUresult e = cuStreamDestroy(stream);
    return (int)(e ? e : cuGreenCtxDestroy(ctx));
}
